// Host engine and C ABI of libspegg_gb300 (see include/spegg.h).
//
// A population owns one device arena.  Biallelic populations are formed by the
// generation kernel (generations.cuh): alone, in cooperative launches of many
// generations, or as members of a batch or server by teams of blocks (TeamSet).
// Continuous allelic values take two launches per generation, enqueued as a
// cached CUDA graph of kGraphChunk generations.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "spegg.h"
#include "spegg_engine.h"
#include "spegg_internal.h"

namespace spg {

thread_local std::string g_last_error;

int fail(int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_last_error = buf;
    return code;
}

int cuda_fail(cudaError_t e, const char *what) {
    return fail(SPG_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

// ------------------------------------------------------------ host tables
// Binomial(n_copies, mu) CDF in Q32 with IEEE-double basic operations in the
// fixed order stated in spegg.h (each product/quotient rounded separately).
uint32_t mutation_cdf(double mu, uint32_t n_copies, uint32_t *cdf) {
    const double q = 1.0 - mu;
    double p_k = 1.0;
    for (uint32_t i = 0; i < n_copies; ++i) p_k = p_k * q;
    double running = 0.0;
    uint32_t entries = 0;
    for (uint32_t k = 0; k <= n_copies && entries < (uint32_t)kMaxKmax; ++k) {
        running = running + p_k;
        const double q32 = running * 4294967296.0;
        if (q32 >= 4294967295.0) break;
        cdf[entries++] = (uint32_t)q32;
        const double t1 = p_k * (double)(n_copies - k);
        const double t2 = t1 / (double)(k + 1);
        const double t3 = t2 * mu;
        p_k = t3 / q;
    }
    return entries;
}

// Per-locus values in offset binary: v_l - v_min split into bit planes, plane
// b word w holding bit b of the offsets of loci 32w .. 32w+31.
static void offset_planes(const int16_t *v, uint32_t n_loci, uint32_t *planes, int32_t &v_min, uint32_t &nplanes) {
    const uint32_t W = n_loci / 32;
    int32_t lo = v[0], hi = v[0];
    for (uint32_t l = 1; l < n_loci; ++l) {
        lo = std::min<int32_t>(lo, v[l]);
        hi = std::max<int32_t>(hi, v[l]);
    }
    const uint32_t span = (uint32_t)(hi - lo);
    uint32_t np = 0;
    while (np < 32 && (span >> np) != 0u) ++np;
    std::memset(planes, 0, sizeof(uint32_t) * kMaxPlanes * kMaxWords);
    for (uint32_t l = 0; l < n_loci; ++l) {
        const uint32_t off = (uint32_t)((int32_t)v[l] - lo);
        for (uint32_t b = 0; b < np && b < (uint32_t)kMaxPlanes; ++b)
            if ((off >> b) & 1u) planes[b * W + l / 32] |= 1u << (l % 32);
    }
    v_min = lo;
    nplanes = np;
}

// Effects in offset binary (the additive genetic value's bit planes).
void effect_planes(const int16_t *effects, uint32_t n_loci, PopParams &prm) {
    offset_planes(effects, n_loci, prm.planes, prm.e_min, prm.nplanes);
}

// Byte tables of per-locus values v: table
// k, entry b is the sum of v[8k + i] over the bits i set in b -- the value of
// the eight loci 8k .. 8k+7 held in byte k of a haplotype (locus l is bit l % 32
// of word l / 32).  Exact in int32 (at most 8 * 32768 in magnitude).
void byte_tables(const int16_t *v, uint32_t n_loci, int32_t *lut) {
    std::memset(lut, 0, sizeof(int32_t) * kMaxLutBytes * kLutWords);
    for (uint32_t k = 0; k < n_loci / 8; ++k)
        for (uint32_t b = 0; b < (uint32_t)kLutWords; ++b) {
            int32_t sum = 0;
            for (uint32_t i = 0; i < 8; ++i)
                if ((b >> i) & 1u) sum += v[8 * k + i];
            lut[k * kLutWords + b] = sum;
        }
}

// v * 2^s as f16, v of at most 11 significant bits, the result in the normal range.
static uint32_t f16_scaled(int32_t v, int s) {
    if (v == 0) return 0u;
    const uint32_t m = (uint32_t)(v < 0 ? -v : v);
    int e = 0;
    while ((m >> e) > 1u) ++e;  // 2^e <= m < 2^(e+1)
    const uint32_t frac = e > 10 ? (m >> (e - 10)) & 0x3FFu : (m << (10 - e)) & 0x3FFu;
    return (v < 0 ? 0x8000u : 0u) | (uint32_t)(e + s + 15) << 10 | frac;
}

// The B fragments of the generation kernel's products (generations.cuh): lane
// 4n + q holds column n of the element pairs that lane q of a row's group
// makes.  Pair r of a lane: element position p (its bit in the half words,
// after the kernel's shifts) and the loci in its low and high half.  Even
// columns: the value (its low digit), odd columns: the allele count of the
// element (its high digit of radix 2048), each scaled by 2^(4 - p).
void value_fragments(const int16_t *effects, const int16_t *dominance, uint32_t n_loci, ValueFragments &vf,
                     uint32_t &two_digits) {
    const uint32_t W = n_loci / 32, regs = W >= 4 ? 16u : 4u * W, room = std::max(regs, 8u);
    auto value = [&](uint32_t t, uint32_t l) {  // additive; heterozygous, homozygous
        return !dominance ? (int32_t)effects[l] : t == 0 ? effects[l] + (int32_t)dominance[l] : 2 * (int32_t)effects[l];
    };
    two_digits = 0;
    for (uint32_t t = 0; t < (dominance ? 2u : 1u); ++t)
        for (uint32_t l = 0; l < n_loci; ++l)
            if (value(t, l) > 2048 || value(t, l) < -2048) two_digits = 1;
    std::memset(&vf, 0, sizeof vf);
    for (uint32_t t = 0; t < (dominance ? 2u : 1u); ++t)
        for (uint32_t set = 0; set < (W == 8 ? 2u : 1u); ++set)
            for (uint32_t r = 0; r < regs; ++r)
                for (uint32_t lane = 0; lane < 32; ++lane) {
                    const uint32_t q = lane & 3u, odd = (lane >> 2) & 1u;
                    const uint32_t word = W >= 4 ? 4u * set + q : W == 2 ? q & 1u : 0u;
                    const uint32_t part = W >= 4 ? 0u : W == 2 ? 8u * (q >> 1) : 4u * q;  // first bit of the lane's part
                    uint32_t bit, p;
                    if (dominance) {  // one bit per locus
                        bit = r;
                        p = r <= 10 ? r : r - 5;
                    } else {          // two bits per locus: even loci, then odd ones
                        const uint32_t i = r % (regs / 2);
                        bit = 2 * i + r / (regs / 2);
                        p = i <= 5 ? 2 * i : 2 * i - 4;
                    }
                    uint32_t pair = 0;
                    for (uint32_t h = 0; h < 2; ++h) {
                        const int32_t v = value(t, 32u * word + part + bit + 16u * h);
                        const int32_t d0 = two_digits ? ((v + 1024) & 2047) - 1024 : v;
                        const int32_t x = !odd ? d0 : two_digits ? (v - d0) / 2048 : dominance && t == 1 ? 2 : 1;
                        pair |= f16_scaled(x, 4 - (int)p) << (16 * h);
                    }
                    const uint32_t at = dominance ? r : r % (regs / 2) + r / (regs / 2) * (room / 2);
                    vf.table[t][set * room * 32u + (at / 4u) * 128u + lane * 4u + at % 4u] = pair;
                }
}

// Resource factor of the ecology, same arithmetic as the device finalizer.
uint32_t factor_q32_host(double R, double R_half) {
    const double den = R + R_half;
    const double q = R / den;
    const double scaled = q * 4294967296.0;
    if (scaled >= 4294967294.0) return 0xFFFFFFFEu;
    if (!(scaled > 0.0)) return 0u;
    return (uint32_t)scaled;
}

// ----------------------------------------------------------- device memory
void *Allocator::alloc(size_t bytes, cudaStream_t s) const {
    if (hooks.alloc) return hooks.alloc(bytes, hooks.ctx);
    void *p = nullptr;
    if (cudaMallocAsync(&p, bytes, s) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}

void Allocator::release(void *p, cudaStream_t s) const {
    if (!p) return;
    if (hooks.free) hooks.free(p, hooks.ctx);
    else cudaFreeAsync(p, s);
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ----------------------------------------------------------- validation
int validate_desc(const spg_pop_desc *d) {
    if (!d) return fail(SPG_ERR_INVALID, "population description is NULL");
    if (d->n == 0 || d->n > 0x7FFFFFFFu) return fail(SPG_ERR_INVALID, "n must be in [1, 2^31-1] (got %u)", d->n);
    if (!(d->n_loci == 32 || d->n_loci == 64 || d->n_loci == 128 || d->n_loci == 256))
        return fail(SPG_ERR_INVALID, "n_loci must be 32, 64, 128 or 256 (got %u)", d->n_loci);
    if (!d->effects) return fail(SPG_ERR_INVALID, "effects is NULL");
    if (!d->surv_table) return fail(SPG_ERR_INVALID, "surv_table is NULL");
    if (d->bin_shift > 31) return fail(SPG_ERR_INVALID, "bin_shift must be <= 31");
    if (!(d->mu >= 0.0 && d->mu < 1.0)) return fail(SPG_ERR_INVALID, "mu must be in [0, 1)");
    if (d->stats_capacity > (1u << 24)) return fail(SPG_ERR_INVALID, "stats_capacity must be <= 2^24");
    if (d->allele_model > 1u) return fail(SPG_ERR_INVALID, "allele_model must be 0 (biallelic) or 1 (continuous)");
    if (d->allele_model == 1u) {
        if (d->map_morgans || d->mother_weights || d->father_weights || d->dominance || d->init_genotypes)
            return fail(SPG_ERR_INVALID, "continuous allelic values take no linkage map, weights, dominance or "
                                         "init_genotypes (use init_values)");
        if (!(d->mut_sd >= 0.0 && d->mut_sd < 64.0) || !(d->env_sd >= 0.0 && d->env_sd < 64.0))
            return fail(SPG_ERR_INVALID, "mut_sd and env_sd must be in [0, 64)");
    }
    return SPG_OK;
}

int build_params(const spg_pop_desc *d, PopParams &prm) {
    std::memset(&prm, 0, sizeof prm);
    std::memcpy(prm.table, d->surv_table, sizeof prm.table);
    effect_planes(d->effects, d->n_loci, prm);
    if (prm.nplanes > (uint32_t)kMaxPlanes) return fail(SPG_ERR_INVALID, "effects span more than 16 bits");
    if (d->dominance) {
        offset_planes(d->dominance, d->n_loci, prm.dplanes, prm.d_min, prm.ndplanes);
        if (prm.ndplanes > (uint32_t)kMaxPlanes)
            return fail(SPG_ERR_INVALID, "dominance deviations span more than 16 bits");
        for (uint32_t l = 0; l < d->n_loci; ++l) prm.has_dom |= d->dominance[l] != 0 ? 1u : 0u;
    }
    prm.kmax = mutation_cdf(d->mu, 2 * d->n_loci, prm.cdf);
    prm.bias = d->bin_bias;
    prm.shift = d->bin_shift;
    prm.n = d->n;
    prm.n_loci = d->n_loci;
    prm.words = d->n_loci / 32;
    prm.key0 = (uint32_t)(d->seed & 0xFFFFFFFFull);
    prm.key1 = (uint32_t)(d->seed >> 32);
    prm.rep = d->replicate;
    prm.has_eco = 0;
    prm.stats_cap = d->stats_capacity ? d->stats_capacity : 1024u;
    prm.linked = d->map_morgans ? 1u : 0u;
    prm.link = nullptr;  // set once the population's memory exists
    prm.weighted = (d->mother_weights || d->father_weights) ? 1u : 0u;
    prm.weights = nullptr;
    prm.continuous = d->allele_model == 1u ? 1u : 0u;
    prm.s_mut = prm.continuous ? (long long)std::floor(d->mut_sd * 256.0 * 65536.0 + 0.5) : 0;
    prm.s_env = prm.continuous ? (long long)std::floor(d->env_sd * 512.0 * 65536.0 + 0.5) : 0;
    return SPG_OK;
}

// Linkage map (Haldane, no interference): w_l = map distance of the linked
// interval between loci l-1 and l (0 where locus l starts a chromosome),
// D = sum w_l; crossover count CDF = Binomial(kLinkSites, D / kLinkSites);
// interval CDF cum[l] = floor(2^32 * (s / D)) with s the running sum of w.
int build_link(const double *map, uint32_t n_loci, LinkParams &lp) {
    std::memset(&lp, 0, sizeof lp);
    double w[kMaxLoci];
    double D = 0.0;
    uint32_t chrom = 0;
    lp.first[0] = 0;
    w[0] = 0.0;
    for (uint32_t l = 1; l < n_loci; ++l) {
        const double m = map[l];
        if (!(m == m) || std::isinf(m)) return fail(SPG_ERR_INVALID, "map_morgans[%u] is not finite", l);
        if (m < 0.0) {
            if (++chrom >= (uint32_t)kMaxChrom)
                return fail(SPG_ERR_INVALID, "a linkage map holds at most %d chromosomes", kMaxChrom);
            lp.first[chrom] = (uint16_t)l;
            w[l] = 0.0;
        } else {
            w[l] = m;
        }
        D = D + w[l];
    }
    lp.nchrom = chrom + 1;
    if (!(D <= kMaxMapMorgans)) return fail(SPG_ERR_INVALID, "the linkage map is longer than 16 Morgans");
    lp.kmax = mutation_cdf(D / (double)kLinkSites, kLinkSites, lp.cdf);
    double run = 0.0;
    for (uint32_t l = 0; l < n_loci; ++l) {
        if (D > 0.0) {
            run = run + w[l];
            const double x = (run / D) * 4294967296.0;
            lp.cum[l] = x >= 4294967295.0 ? 0xFFFFFFFFu : (uint32_t)x;
        } else {
            lp.cum[l] = 0;
        }
    }
    // guide[h]: the interval of the bucket's first uniform and the interval
    // boundaries inside the bucket (none for most buckets: the guide entry is
    // the answer)
    constexpr uint32_t shift = 32u - (uint32_t)kLinkGuideBits;
    auto interval = [&](uint32_t u) {
        uint32_t I = 0;
        while (I + 1 < n_loci && lp.cum[I] <= u) ++I;
        return I;
    };
    for (uint32_t h = 0; h < (uint32_t)kLinkGuide; ++h) {
        const uint32_t lo = h << shift, hi = lo | ((1u << shift) - 1u);
        const uint32_t I0 = interval(lo), nb = std::min<uint32_t>(interval(hi) - I0, 2u);
        lp.guide[h] = I0 | (nb << 26);
    }
    return SPG_OK;
}

// Weighted parents: t[b] = floor(2^32 * w[b] / max w) (integer arithmetic),
// 0xFFFFFFFF where w[b] is the maximum; a NULL table is uniform.
static int weight_thresholds(const uint32_t *w, uint32_t *acc, const char *role) {
    if (!w) {
        for (int b = 0; b < kBins; ++b) acc[b] = kCertain;
        return SPG_OK;
    }
    uint32_t mx = 0;
    for (int b = 0; b < kBins; ++b) mx = std::max(mx, w[b]);
    if (mx == 0) return fail(SPG_ERR_INVALID, "%s weights are all zero", role);
    for (int b = 0; b < kBins; ++b)
        acc[b] = w[b] == mx ? kCertain : (uint32_t)(((uint64_t)w[b] << 32) / mx);
    return SPG_OK;
}

int build_weights(const uint32_t *mother_w, const uint32_t *father_w, WeightParams &wp) {
    int rc = weight_thresholds(mother_w, wp.acc[0], "mother");
    if (rc == SPG_OK) rc = weight_thresholds(father_w, wp.acc[1], "father");
    return rc;
}

// ------------------------------------------------------------ population
uint32_t bucket_count(uint32_t n) { return (n + kBucket - 1) / kBucket; }

// The arena of a population of continuous allelic values.
PopLayout layout_for(uint32_t n, uint32_t words, uint32_t nbuckets, uint32_t cap) {
    PopLayout L{};
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off = align_up(off + bytes, 256);
        return at;
    };
    L.params = take(sizeof(PopParams));
    L.state = take(sizeof(DevState));
    L.ring = take((size_t)cap * sizeof(spg_stats));
    L.acc = take(sizeof(StatAcc) * kAccCopies);
    L.geno0 = take((size_t)n * 2 * words * 4);
    L.geno1 = take((size_t)n * 2 * words * 4);
    L.surv0 = take((size_t)n * 4);
    L.surv1 = take((size_t)n * 4);
    L.alive = take((size_t)nbuckets * kBucketWords * 4);
    L.buckets = take((size_t)2 * nbuckets * 4);
    L.segment = take(sizeof(Segment));
    L.total = off;
    return L;
}

// Slots of a single population: at most kMaxSlots of whole groups of 32, or
// one per warp of a block for a population that one block forms.
uint32_t slot_length(uint32_t n) {
    const uint64_t slots = n <= 32u * kOneBlockGroups ? kSoloThreads / 32u : kMaxSlots;
    return (uint32_t)(((uint64_t)n + 32ull * slots - 1) / (32ull * slots));
}
uint32_t slot_count(uint32_t n) {
    const uint32_t len = 32u * slot_length(n);
    return (uint32_t)(((uint64_t)n + len - 1) / len);
}

// The arena of a single biallelic population (generations.cuh): one buffer
// of full records, two of packed survivors.
PopLayout solo_layout_for(uint32_t n, uint32_t words, uint32_t cap, bool weighted) {
    PopLayout L{};
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off = align_up(off + bytes, 256);
        return at;
    };
    L.solo = true;
    L.params = take(sizeof(PopParams));
    L.state = take(sizeof(DevState));
    L.ring = take((size_t)cap * sizeof(spg_stats));
    L.acc = take(sizeof(StatAcc) * kAccCopies);
    L.geno0 = L.geno1 = take((size_t)n * 2 * words * 4);
    for (size_t &x : L.packed) x = take((size_t)n * 2 * words * 4);
    L.surv0 = L.surv1 = take((size_t)n * 4);
    L.alive = take(((size_t)n + 31) / 32 * 4);
    for (size_t &x : L.counts) x = take((size_t)slot_count(n) * 4);
    L.gen_acc = take(sizeof(GenAcc) * 3 * kGenAccCopies);
    L.barrier = take(sizeof(unsigned long long));
    L.frag = take(sizeof(ValueFragments));
    L.link = take(sizeof(LinkParams));
    L.weighted = weighted;
    if (weighted) {
        L.weights = take(sizeof(WeightParams));
        for (size_t &x : L.mate) x = take((size_t)n * 8);
    }
    L.total = off;
    return L;
}

// The generation kernel's arguments for a population at v (solo layout); the
// fragments' flags (dom, two_digits) are already in a.
void solo_args(const PopView &v, const PopParams &prm, SoloArgs &a) {
    a.prm = reinterpret_cast<const PopParams *>(v.base + v.L.params);
    a.frag = reinterpret_cast<const ValueFragments *>(v.base + v.L.frag);
    for (uint32_t i = 0; i < 2; ++i) {
        a.packed[i] = reinterpret_cast<uint32_t *>(v.base + v.L.packed[i]);
        a.counts[i] = reinterpret_cast<uint32_t *>(v.base + v.L.counts[i]);
        a.mate[i] = v.L.weighted ? reinterpret_cast<uint2 *>(v.base + v.L.mate[i]) : nullptr;
    }
    a.geno = reinterpret_cast<uint32_t *>(v.base + v.L.geno0);
    a.alive = reinterpret_cast<uint32_t *>(v.base + v.L.alive);
    a.surv = reinterpret_cast<uint32_t *>(v.base + v.L.surv0);
    a.state = reinterpret_cast<DevState *>(v.base + v.L.state);
    a.acc = reinterpret_cast<GenAcc *>(v.base + v.L.gen_acc);
    a.barrier = reinterpret_cast<unsigned long long *>(v.base + v.L.barrier);
    a.ring = reinterpret_cast<spg_stats *>(v.base + v.L.ring);
    for (uint32_t i = 0; i < 10; ++i) {
        a.keys[2 * i] = prm.key0 + i * 0x9E3779B9u;
        a.keys[2 * i + 1] = prm.key1 + i * 0xBB67AE85u;
    }
    a.barrier_tries = kBarrierTries;
    a.words = prm.words;
    a.rep = prm.rep;
    a.kmax = prm.kmax;
    a.mut_from = prm.kmax ? prm.cdf[0] : 0xFFFFFFFFu;
    a.shift = prm.shift;
    a.bias = prm.bias;
    a.narrow_bias = prm.bias < (1 << 30) && prm.bias > -(1 << 30) ? 1u : 0u;  // |genetic value| < 2^26
    a.stats_cap = v.cap;
    a.n = v.n;
    a.slot_len = slot_length(v.n);
    a.nslots = slot_count(v.n);
    a.guide_bits = 2;  // four to eight entries per slot
    while ((a.nslots >> (a.guide_bits - 2)) != 0u && a.guide_bits < (uint32_t)kMaxGuideBits) ++a.guide_bits;
    a.has_eco = prm.has_eco;
    a.eco_model = prm.eco_model;
    a.eco_r = prm.r;
    a.eco_r_sd = prm.r_sd;
    a.eco_K = prm.K;
    a.eco_R_half = prm.R_half;
}

// Least warps of work per block: a small population takes as few SMs as give
// every one of them this many warps (at 10,000 offspring 4 and 16 warps differ
// by less than the barrier does).
constexpr uint32_t kSoloMinWarps = 4;

uint32_t most_blocks(uint32_t n, uint32_t resident) {
    return n <= 32u * kOneBlockGroups ? 1u : std::max(1u, std::min(resident, slot_count(n) / kSoloMinWarps));
}

// Blocks of a population alone: a block fills an SM, so populations on streams of
// their own run at the same time only when their blocks fit together.  A small
// one therefore takes half of what the device holds at most while that is ten
// slots a block or less: 200 generations of one, two and four populations of 10^4,
// ms: 0.95 / 1.88 / 3.75 with 78 blocks, 0.95 / 0.96 / 1.90 with 76 (a quarter:
// 0.99 / 0.99 / 1.00), of 2 x 10^4 1.04 / 2.07 / 4.10 and 1.06 / 1.07 / 2.11; before
// the generation kernel 1.66 / 1.64 / 1.78 and 1.80 / 1.93 / 2.20.  With 16 slots a
// block one alone takes a fifth longer.  At L = 256 the line is at five slots (2 x
// 10^4 alone: 6.9 us a generation on all blocks, 7.2 on half).
uint32_t solo_grid(uint32_t n, uint32_t words, uint32_t resident) {
    const uint32_t blocks = most_blocks(n, resident), half = std::max(resident / 2u, 1u);
    return slot_count(n) <= (words == 8u ? 5u : 10u) * half ? std::min(blocks, half) : blocks;
}

// ------------------------------------------------------------ teams
// Cycles of a generation on k blocks of 16 warps: closing it alone or with a
// barrier, and rounds of the warps' groups (measured, L = 32 .. 256; a linkage
// map, parent weights and general values make a round longer: 10^6 x 128 takes
// 75, 48 and 31 us a generation, plain 26).
static double round_cycles(const TeamMember &m) {
    const double plain = m.words == 1 ? 2000.0 : m.words == 2 ? 2300.0 : m.words == 4 ? 3100.0 : 5400.0;
    return plain * (m.linked ? 3.0 : 1.0) * (m.weighted ? 1.9 : 1.0) * (m.general ? 1.2 : 1.0);
}
TeamMember team_member(const SoloArgs &a, bool linked, bool weighted) {
    TeamMember m;
    m.args = &a;
    m.n = a.n;
    m.words = a.words;
    m.linked = linked;
    m.weighted = weighted;
    m.general = a.dom || a.two_digits || !a.narrow_bias;
    return m;
}
static double block_work(const TeamMember &m) { return ((double)m.n + 31.0) / 32.0 / 16.0 * round_cycles(m); }
static double team_cycles(const TeamMember &m, uint32_t k) {
    const double groups = ((double)m.n + 31.0) / 32.0;
    return (k == 1 ? 6000.0 : 11000.0) + std::max(1.0, groups / (16.0 * k)) * round_cycles(m);
}

// Generations of one launch of a population on `blocks` of the device's blocks:
// other streams' work waits for a launch that fills the device, so it is cut at
// about 1.5 ms (at eight generations at least; a launch costs about 6 us more than
// its generations, 26.0 -> 26.1 us a generation at 10^6 x 128).  A call of one
// generation of 1,000 offspring beside 1,000 generations of 10^6 x 128 waited 13.5
// ms with launches of 512, and 1.5 now.  Beside a launch of half the device or
// less there is room (512 generations of it are some 2.5 ms).
constexpr double kLaunchCycles = 3.0e6;
uint32_t launch_generations(const TeamMember &m, uint32_t blocks, uint32_t resident) {
    if (2u * blocks <= resident) return kSoloLaunchGens;
    return (uint32_t)std::min<double>(kSoloLaunchGens, std::max(8.0, kLaunchCycles / team_cycles(m, blocks)));
}

// Blocks below which all teams' records together would not stay in L2: with
// every block at its share of such a member, parents and survivors (16 W bytes
// an individual) come to kTeamL2Bytes (152 members of 60,000 x 128 loci on a
// block each formed an individual in 35 ps, of 30,000 in 25).
constexpr double kTeamL2Bytes = 2.5e8;
static double resident_blocks(const TeamMember &m, uint32_t blocks) {
    return std::ceil(16.0 * m.words * m.n / (kTeamL2Bytes / blocks));
}

// Teams for the members on `blocks` blocks: by locus count (the order in which
// k_teams takes them), the longest first, each with as
// many blocks as keep it below a share of the whole and its records in L2, on
// the blocks that are free soonest; the share that gives the shortest schedule
// is kept.  All blocks have their teams in the members' one order (k_teams).
// Returns the estimated cycles of a generation of all members.
double schedule_teams(const std::vector<TeamMember> &members, uint32_t blocks, std::vector<TeamPlace> &places,
                      std::vector<uint32_t> &block_places) {
    const uint32_t M = (uint32_t)members.size();
    std::vector<uint32_t> order(M);
    std::vector<double> work(M);
    double total = 0.0;
    for (uint32_t m = 0; m < M; ++m) {
        order[m] = m;
        work[m] = block_work(members[m]);
        total += work[m];
    }
    std::stable_sort(order.begin(), order.end(), [&](uint32_t x, uint32_t y) {
        return members[x].words != members[y].words ? members[x].words > members[y].words : work[x] > work[y];
    });
    // places of a schedule in the members' order, with their blocks
    struct Dealt {
        uint32_t block;
        TeamPlace place;
    };
    double best = -1.0;
    std::vector<Dealt> kept, dealt;
    std::vector<double> free_at;
    std::vector<uint32_t> by_time;
    // (a little above one: members that divide the blocks without rounding up to
    // one block too many, which would put them one after the other; the same for
    // more members than blocks)
    for (const double share : {0.1, 0.15, 0.25, 0.4, 0.6, 1.0, 1.06, 1.25, 1.6}) {
        if (share > 1.0 && M > blocks) break;
        free_at.assign(blocks, 0.0);
        by_time.resize(blocks);
        for (uint32_t b = 0; b < blocks; ++b) by_time[b] = b;
        dealt.clear();
        double end = 0.0;
        for (const uint32_t m : order) {
            const double want = std::max(std::ceil(work[m] / (share * total / blocks)), resident_blocks(members[m], blocks));
            const uint32_t k = (uint32_t)std::max(1.0, std::min<double>(want, most_blocks(members[m].n, blocks)));
            if (k == 1u) {  // (most members of a large batch: a plain search is quicker)
                const size_t b = (size_t)(std::min_element(free_at.begin(), free_at.end()) - free_at.begin());
                free_at[b] += team_cycles(members[m], 1u);
                dealt.push_back(Dealt{(uint32_t)b, TeamPlace{m, 0u, 1u}});
                end = std::max(end, free_at[b]);
                continue;
            }
            std::nth_element(by_time.begin(), by_time.begin() + (k - 1), by_time.end(),
                             [&](uint32_t x, uint32_t y) { return free_at[x] != free_at[y] ? free_at[x] < free_at[y] : x < y; });
            double start = 0.0;
            for (uint32_t i = 0; i < k; ++i) start = std::max(start, free_at[by_time[i]]);
            const double done = start + team_cycles(members[m], k);
            for (uint32_t i = 0; i < k; ++i) {
                free_at[by_time[i]] = done;
                dealt.push_back(Dealt{by_time[i], TeamPlace{m, (uint16_t)i, (uint16_t)k}});
            }
            end = std::max(end, done);
        }
        if (best < 0.0 || end < best) {
            best = end;
            kept.swap(dealt);
        }
    }
    // by block, each block's in the members' order
    block_places.assign(blocks + 1u, 0u);
    for (const Dealt &d : kept) ++block_places[d.block + 1u];
    for (uint32_t b = 0; b < blocks; ++b) block_places[b + 1u] += block_places[b];
    places.resize(kept.size());
    std::vector<uint32_t> at(block_places.begin(), block_places.end() - 1);
    for (const Dealt &d : kept) places[at[d.block]++] = d.place;
    return std::max(best, 0.0);
}

// SM cycles of a generation of continuous values beside teams, and the SMs it
// fills: four blocks of 256 each.  Half of what it takes alone (92, 143, 234 and 472
// us at N = 10^6 for L = 32 .. 256): much of that waits for memory, which more SMs
// do not shorten (two members of 2 x 10^5, one of them continuous, 36.4 us a
// generation with all of it, 29.7 with half).
double continuous_work(uint32_t n, uint32_t n_loci) {
    return (double)n * (n_loci == 32 ? 14.5 : n_loci == 64 ? 22.5 : n_loci == 128 ? 37.0 : 74.0);
}
uint32_t continuous_blocks(uint32_t n) { return (uint32_t)(((uint64_t)n + 1023u) / 1024u); }

// `blocks` blocks dealt to several kinds by their work, each at least one and at
// most as many as it can use.
std::vector<uint32_t> deal_blocks(const std::vector<double> &work, const std::vector<uint32_t> &most, uint32_t blocks) {
    std::vector<uint32_t> got(work.size(), 0u);
    uint32_t left = blocks;
    for (size_t k = 0; k < work.size(); ++k)
        if (work[k] > 0.0 && left) {
            got[k] = 1u;
            --left;
        }
    for (; left; --left) {  // the next block to the kind with the most work per block
        size_t next = work.size();
        for (size_t k = 0; k < work.size(); ++k)
            if (got[k] && got[k] < most[k] && (next == work.size() || work[k] * got[next] > work[next] * got[k])) next = k;
        if (next == work.size()) break;
        ++got[next];
    }
    return got;
}

// Kinds need kernels of their own (bodies of all kinds in one kernel take minutes
// to compile and spill), and a launch of a kind with few members leaves most
// blocks idle.  So the blocks are dealt to the kinds and their launches run side
// by side, unless the kinds one after the other, each on all blocks, are
// estimated to be faster.
int TeamSet::build(const std::vector<TeamMember> &all, const Allocator &alloc, cudaStream_t stream, bool singles,
                   double kept, uint32_t kept_blocks) {
    std::vector<double> work(kTeamKinds + 1u, 0.0);
    std::vector<uint32_t> most(kTeamKinds + 1u, 0u);
    uint32_t kinds = 0, resident = 0;
    for (TeamLaunch &t : launch) t.members.clear();
    // plain members join the general ones (whose kernel is 4 % slower for them, but
    // a launch less: calls of one generation of two members of 10^4 10.8 us
    // against 16.6) unless they are most of the work
    double plain = 0.0, general = 0.0;
    for (const TeamMember &m : all)
        if (team_kind(m.linked, m.weighted, m.general) <= 1u) (m.general ? general : plain) += block_work(m);
    const bool join = general > 0.0 && plain <= 8.0 * general;
    for (const TeamMember &m : all) launch[team_kind(m.linked, m.weighted, m.general || join)].members.push_back(m);
    for (uint32_t kind = 0; kind < kTeamKinds; ++kind) {
        TeamLaunch &t = launch[kind];
        if (t.members.empty()) continue;
        if (!t.kernel.fn) {
            t.kernel = team_kernel(kind);
            const int rc = prepare_solo(t.kernel);
            if (rc != SPG_OK) return fail(rc, "team kernel setup failed");
        }
        ++kinds;
        resident = resident ? std::min(resident, t.kernel.resident) : t.kernel.resident;
        for (const TeamMember &m : t.members) {
            work[kind] += block_work(m);
            most[kind] = std::min(t.kernel.resident, most[kind] + most_blocks(m.n, t.kernel.resident));
        }
    }
    work[kTeamKinds] = kept;
    most[kTeamKinds] = kept_blocks;
    const std::vector<uint32_t> dealt = deal_blocks(work, most, resident);
    const uint32_t mine = resident - (kinds ? std::min(dealt[kTeamKinds], resident - 1u) : 0u);
    std::vector<TeamPlace> places[2][kTeamKinds];
    std::vector<uint32_t> starts[2][kTeamKinds];
    double cycles[2][kTeamKinds] = {}, total[2] = {0.0, 0.0};  // one after the other, side by side
    for (uint32_t kind = 0; kind < kTeamKinds; ++kind) {
        const TeamLaunch &t = launch[kind];
        if (t.members.empty()) continue;
        cycles[0][kind] = schedule_teams(t.members, mine, places[0][kind], starts[0][kind]);
        total[0] += cycles[0][kind];
        if (kinds > 1u && kinds <= mine) {
            cycles[1][kind] = schedule_teams(t.members, dealt[kind], places[1][kind], starts[1][kind]);
            total[1] = std::max(total[1], cycles[1][kind]);
        }
    }
    beside = kinds > 1u && kinds <= mine && total[1] < total[0];
    if (beside && !forked && cudaEventCreateWithFlags(&forked, cudaEventDisableTiming) != cudaSuccess)
        return fail(SPG_ERR_CUDA, "cudaEventCreate");
    // bitmap words that a block lists of a one-generation call: about eight blocks
    // per SM, 64 words at least
    uint64_t words = 0;
    for (const TeamMember &m : all) words += (m.n + 31u) / 32u;
    const uint64_t per_part = std::max<uint64_t>(64u, words / (8ull * std::max(resident, 1u)));
    std::vector<ClosePart> part_list;
    std::vector<SoloArgs> args[kTeamKinds];
    uint32_t first = kTeamKinds;  // stays on the caller's stream
    for (uint32_t kind = 0; kind < kTeamKinds; ++kind) {
        TeamLaunch &t = launch[kind];
        if (t.members.empty()) continue;
        first = std::min(first, kind);
        const std::vector<TeamPlace> &place = places[beside ? 1 : 0][kind];
        const std::vector<uint32_t> &start = starts[beside ? 1 : 0][kind];
        t.blocks = beside ? dealt[kind] : mine;
        t.cycles = cycles[beside ? 1 : 0][kind];
        if (beside && first != kind && !t.side) {
            cudaError_t e = cudaStreamCreateWithFlags(&t.side, cudaStreamNonBlocking);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&t.joined, cudaEventDisableTiming);
            if (e != cudaSuccess) return cuda_fail(e, "team streams");
        }
        const size_t o_places = align_up(t.members.size() * sizeof(SoloArgs), 256),
                     o_blocks = align_up(o_places + place.size() * sizeof(TeamPlace), 256),
                     need = o_blocks + start.size() * 4;
        if (need > t.capacity) {
            if (t.table) alloc.release(t.table, stream);
            t.capacity = 2 * need;  // (a server's set changes)
            t.table = static_cast<char *>(alloc.alloc(t.capacity, stream));
            if (!t.table) {
                t.capacity = 0;
                return fail(SPG_ERR_OOM, "team table allocation failed");
            }
        }
        for (const TeamMember &m : t.members) {
            SoloArgs a = *m.args;
            a.close_slots = (uint32_t)std::min<uint64_t>(256u, (per_part + a.slot_len - 1u) / a.slot_len);
            for (uint32_t i = 0; singles && i * a.close_slots < a.nslots; ++i)
                part_list.push_back(ClosePart{reinterpret_cast<const SoloArgs *>(t.table) + args[kind].size(), i, 0u});
            args[kind].push_back(a);
        }
        cudaError_t e = cudaMemcpyAsync(t.table, args[kind].data(), args[kind].size() * sizeof(SoloArgs),
                                        cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(t.table + o_places, place.data(), place.size() * sizeof(TeamPlace), cudaMemcpyHostToDevice,
                                stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(t.table + o_blocks, start.data(), start.size() * 4, cudaMemcpyHostToDevice, stream);
        if (e != cudaSuccess) return cuda_fail(e, "upload team table");
        t.args.members = reinterpret_cast<const SoloArgs *>(t.table);
        t.args.places = reinterpret_cast<const TeamPlace *>(t.table + o_places);
        t.args.block_places = reinterpret_cast<const uint32_t *>(t.table + o_blocks);
    }
    nparts = (uint32_t)part_list.size();
    if (nparts * sizeof(ClosePart) > parts_capacity) {
        alloc.release(parts, stream);
        parts_capacity = 2 * nparts * sizeof(ClosePart);
        parts = static_cast<ClosePart *>(alloc.alloc(parts_capacity, stream));
        if (!parts) {
            parts_capacity = 0;
            return fail(SPG_ERR_OOM, "team table allocation failed");
        }
    }
    cudaError_t e = nparts ? cudaMemcpyAsync(parts, part_list.data(), nparts * sizeof(ClosePart), cudaMemcpyHostToDevice, stream)
                           : cudaSuccess;
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);  // the host tables go away
    return e == cudaSuccess ? SPG_OK : cuda_fail(e, "upload team table");
}

// A member's changed arguments (its place in the tables stays), in stream order.
int TeamSet::update(const SoloArgs *args, cudaStream_t stream) {
    for (TeamLaunch &t : launch)
        for (size_t i = 0; i < t.members.size(); ++i)
            if (t.members[i].args == args) {
                // (but not close_slots, which only the table holds)
                const cudaError_t e = cudaMemcpyAsync(t.table + i * sizeof(SoloArgs), args, offsetof(SoloArgs, close_slots),
                                                      cudaMemcpyHostToDevice, stream);
                return e == cudaSuccess ? SPG_OK : cuda_fail(e, "update team table");
            }
    return SPG_OK;
}

static cudaError_t launch_early(const void *fn, uint32_t blocks, uint32_t threads, uint32_t smem, void **params,
                                cudaStream_t stream) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, fn, params);
}

// n_gen generations of every member.  A launch is cut at about a quarter of a
// second, so that a team's blocks never wait long for one another.  A call of one
// generation forms it without barriers, and one more launch closes it for all
// members (64, 256 and 4,096 replicates: 77.5, 269 and 3,779 us a call with the
// barriers, 74.6, 258 and 3,717 without).
int TeamSet::step(uint32_t n_gen, bool keep_last, cudaStream_t stream) {
    const bool single = n_gen == 1u && nparts != 0u;
    cudaError_t e = beside ? cudaEventRecord(forked, stream) : cudaSuccess;
    bool first = true;  // the first kind stays on the caller's stream
    for (TeamLaunch &t : launch) {
        if (t.members.empty()) continue;
        cudaStream_t s = beside && !first ? t.side : stream;
        if (e == cudaSuccess && s != stream) e = cudaStreamWaitEvent(s, forked, 0);
        const uint32_t most = (uint32_t)std::max(1.0, std::min<double>(kSoloLaunchGens, 5e8 / std::max(1.0, t.cycles)));
        for (uint32_t done = 0; done < n_gen && e == cudaSuccess;) {
            TeamArgs a = t.args;
            a.n_gen = std::min(n_gen - done, most);
            a.single = single ? 1u : 0u;
            done += a.n_gen;
            a.keep_last = keep_last && done == n_gen ? 1u : 0u;
            void *params[] = {&a};
            e = single ? launch_early(t.kernel.fn, t.blocks, kSoloThreads, t.kernel.smem, params, s)
                       : cudaLaunchCooperativeKernel(t.kernel.fn, dim3(t.blocks), dim3(kSoloThreads), params, t.kernel.smem, s);
        }
        if (e == cudaSuccess && s != stream) e = cudaEventRecord(t.joined, s);
        if (e != cudaSuccess) return cuda_fail(e, "team launch");
        first = false;
    }
    first = true;
    for (TeamLaunch &t : launch) {
        if (!beside || t.members.empty()) continue;
        if (!first && (e = cudaStreamWaitEvent(stream, t.joined, 0)) != cudaSuccess) return cuda_fail(e, "join teams");
        first = false;
    }
    if (single) {
        void *params[] = {&parts};
        e = launch_early(close_members_kernel(), nparts, kCloseThreads, 0u, params, stream);
        if (e != cudaSuccess) return cuda_fail(e, "close launch");
    }
    return SPG_OK;
}

void TeamLaunch::release(const Allocator &alloc, cudaStream_t stream) {
    if (table) alloc.release(table, stream);
    if (side) {
        cudaStreamSynchronize(side);  // (a launch that an error left unjoined)
        cudaStreamDestroy(side);
    }
    if (joined) cudaEventDestroy(joined);
    table = nullptr;
    capacity = 0;
    side = nullptr;
    joined = nullptr;
}

void TeamSet::release(const Allocator &alloc, cudaStream_t stream) {
    for (TeamLaunch &t : launch) t.release(alloc, stream);
    alloc.release(parts, stream);
    parts = nullptr;
    parts_capacity = 0;
    if (forked) cudaEventDestroy(forked);
    forked = nullptr;
}

Segment segment_at(char *base, const PopLayout &L, uint32_t n, uint32_t ntiles, uint32_t tile_begin,
                   uint32_t nbuckets, uint32_t bucket_begin) {
    Segment s{};
    s.n = n;
    s.acc = reinterpret_cast<StatAcc *>(base + L.acc);
    s.prm = reinterpret_cast<const PopParams *>(base + L.params);
    s.geno[0] = reinterpret_cast<uint32_t *>(base + L.geno0);
    s.geno[1] = reinterpret_cast<uint32_t *>(base + L.geno1);
    s.surv[0] = reinterpret_cast<uint32_t *>(base + L.surv0);
    s.surv[1] = reinterpret_cast<uint32_t *>(base + L.surv1);
    s.alive = reinterpret_cast<uint32_t *>(base + L.alive);
    s.bucket_sum = reinterpret_cast<uint32_t *>(base + L.buckets);
    s.state = reinterpret_cast<DevState *>(base + L.state);
    s.ring = reinterpret_cast<spg_stats *>(base + L.ring);
    s.tile_begin = tile_begin;
    s.ntiles = ntiles;
    s.bucket_begin = bucket_begin;
    s.nbuckets = nbuckets;
    return s;
}

// Launch shapes the batch autotuner times, per locus count: threads per
// block x offspring per thread for L <= 64, threads per block x lanes per
// offspring for L >= 128.
Shape autotune_candidate(uint32_t words, uint32_t c) {
    static const uint32_t narrow[kAutotuneCandidates][3] = {{128, 1, 1}, {128, 2, 1}, {256, 1, 1},
                                                             {256, 2, 1}, {512, 1, 1}, {512, 2, 1}};
    static const uint32_t wide[kAutotuneCandidates][3] = {{128, 1, 1}, {256, 1, 1}, {512, 1, 1},
                                                           {128, 1, 2}, {256, 1, 2}, {512, 1, 2}};
    const uint32_t(&e)[3] = words >= 4 ? wide[c % kAutotuneCandidates] : narrow[c % kAutotuneCandidates];
    Shape s;
    s.block = e[0];
    s.items = e[1];
    s.lanes = e[2];
    return s;
}

// A caller's launch shape: 0 fields take the defaults of the locus count.
// words 0: the continuous-allele kernel (256 threads, one offspring each).
int shape_from_abi(uint32_t words, const spg_launch_shape *in, Shape &out) {
    if (words == 0) {
        out = Shape{(uint32_t)kBlock, 1u, 1u};
        if ((in->threads_per_block && in->threads_per_block != (uint32_t)kBlock) ||
            (in->items_per_thread && in->items_per_thread != 1u) ||
            (in->lanes_per_offspring && in->lanes_per_offspring != 1u))
            return fail(SPG_ERR_INVALID, "continuous allelic values run 256 threads, one offspring each");
        return SPG_OK;
    }
    out = default_shape(words);
    if (in->threads_per_block) out.block = in->threads_per_block;
    if (in->lanes_per_offspring) out.lanes = in->lanes_per_offspring;
    out.items = in->items_per_thread ? in->items_per_thread : 1u;
    if (!supported_shape(words, out))
        return fail(SPG_ERR_INVALID,
                    "unsupported launch shape (%u threads, %u offspring per thread, %u lanes per offspring) for %u "
                    "loci: threads 128, 256 or 512; L <= 64: 1 lane, 1 or 2 offspring per thread; L >= 128: 1 or 2 "
                    "lanes, 1 offspring",
                    out.block, out.items, out.lanes, 32u * words);
    return SPG_OK;
}

Shape default_shape(uint32_t words) {
    Shape s;
    s.block = 256;
    s.items = 1;
    s.lanes = words == 8 ? 2u : 1u;  // L = 256: a lane per parent record (two records do not fit a thread)
    return s;
}

GraphChain::~GraphChain() { reset(); }

void GraphChain::reset() {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    exec = nullptr;
    graph = nullptr;
    length = 0;
}

// The launches of a generation kernel: grid, block, shared memory, and
// whether it may start while its predecessor finishes (programmatic
// dependent launch: the kernel waits with griddepcontrol.wait before reading
// the predecessor's results).  The continuous-allele kernel does not.
namespace {
struct KernelLaunch {
    void *fn;
    dim3 grid, block;
    unsigned smem;
    bool programmatic;
};
KernelLaunch offspring_launch(const GenLaunch &gl) {
    return {reinterpret_cast<void *>(gl.offspring.fn), dim3(gl.blocks), dim3(kBlock), gl.offspring.smem,
            gl.offspring.programmatic};
}
KernelLaunch compact_launch(const GenLaunch &gl) {
    return {reinterpret_cast<void *>(gl.compact), dim3(gl.buckets), dim3(kCompactThreads), 0u, true};
}
}  // namespace

int add_generation_nodes(cudaGraph_t graph, const GenLaunch &gl, void **params, uint32_t len) {
    cudaGraphNode_t prev = nullptr;
    for (uint32_t i = 0; i < 2u * len; ++i) {
        const KernelLaunch k = i % 2u == 0 ? offspring_launch(gl) : compact_launch(gl);
        cudaGraphNodeParams np{};
        np.type = cudaGraphNodeTypeKernel;
        np.kernel.func = k.fn;
        np.kernel.gridDim = k.grid;
        np.kernel.blockDim = k.block;
        np.kernel.sharedMemBytes = k.smem;
        np.kernel.kernelParams = params;  // argument values are copied into the nodes
        cudaGraphEdgeData edge{};
        if (k.programmatic) {
            edge.from_port = cudaGraphKernelNodePortProgrammatic;
            edge.type = cudaGraphDependencyTypeProgrammatic;
        }
        cudaGraphNode_t node;
        const cudaError_t e = cudaGraphAddNode(&node, graph, prev ? &prev : nullptr, prev ? &edge : nullptr,
                                               prev ? 1 : 0, &np);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphAddNode");
        prev = node;
    }
    return SPG_OK;
}

// A graph of `len` generations: offspring -> compaction -> offspring -> ...
int GraphChain::build(const GenLaunch &gl, uint32_t len) {
    reset();
    cudaError_t e = cudaGraphCreate(&graph, 0);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGraphCreate");
    GenArgs a = gl.args;
    void *params[] = {&a};
    const int rc = add_generation_nodes(graph, gl, params, len);
    if (rc != SPG_OK) {
        reset();
        return rc;
    }
    e = cudaGraphInstantiate(&exec, graph, 0);
    if (e != cudaSuccess) {
        reset();
        return cuda_fail(e, "cudaGraphInstantiate");
    }
    length = len;
    return SPG_OK;
}

int launch_generation(const GenLaunch &gl, cudaStream_t stream) {
    GenArgs a = gl.args;
    void *params[] = {&a};
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaError_t e = cudaSuccess;
    for (uint32_t step = 0; step < 2u; ++step) {
        const KernelLaunch k = step == 0 ? offspring_launch(gl) : compact_launch(gl);
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = k.grid;
        cfg.blockDim = k.block;
        cfg.dynamicSmemBytes = k.smem;
        cfg.stream = stream;
        cfg.attrs = &attr;
        cfg.numAttrs = k.programmatic ? 1u : 0u;
        e = cudaLaunchKernelExC(&cfg, k.fn, params);
        if (e != cudaSuccess) break;
    }
    return e == cudaSuccess ? SPG_OK : cuda_fail(e, "generation launch");
}

int enqueue_generations(const GenLaunch &gl, uint32_t n_gen, GraphChain &chain, cudaStream_t stream) {
    if (n_gen == 0 || gl.blocks == 0) return SPG_OK;
    if (n_gen >= kGraphChunk) {
        if (!chain.exec) {
            const int rc = chain.build(gl, kGraphChunk);
            if (rc != SPG_OK) return rc;
        }
        for (uint32_t i = 0; i + kGraphChunk <= n_gen; i += kGraphChunk) {
            const cudaError_t e = cudaGraphLaunch(chain.exec, stream);
            if (e != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch");
        }
    }
    for (uint32_t i = 0; i < n_gen % kGraphChunk; ++i) {
        const int rc = launch_generation(gl, stream);
        if (rc != SPG_OK) return rc;
    }
    return SPG_OK;
}

// ------------------------------------------------- launch groups
// Bytes of a launch group's table: segments, the bucket map and the tile map.
size_t group_table_bytes(uint32_t members, uint64_t offspring, uint32_t buckets) {
    return align_up((size_t)members * sizeof(Segment), 256) + align_up((size_t)buckets * 4, 256) +
           align_up((size_t)(offspring / kBlock + members + 1) * 4, 256);
}

// Runs of a launch group (see GenArgs): the members' tiles, in member order,
// with one unit of set-up (tables, pipeline start) before each member, cut
// into P pieces of equal work dealt round-robin to the G blocks (block b
// forms pieces b, b + G, ...: rounds of G pieces of at least min_piece tiles,
// each round a contiguous window of the member list, so the populations being
// formed at any moment are few and their parent records stay in L2 -- the
// flattened replicate loop of Fig. S5 B, scheduled for locality).  A piece is
// one run per member it touches, so every block's work is within a set-up or
// two of the others'.  (Only its test reaches it: teams and tile maps took its
// place.)
void schedule_runs(const std::vector<uint32_t> &tiles, uint32_t G, uint32_t min_piece, std::vector<Run> &runs,
                   std::vector<uint32_t> &block_runs) {
    const uint32_t M = (uint32_t)tiles.size();
    std::vector<uint64_t> ustart(M + 1, 0ull), tstart(M + 1, 0ull);  // prefix units, prefix tiles
    for (uint32_t m = 0; m < M; ++m) {
        ustart[m + 1] = ustart[m] + (tiles[m] ? tiles[m] + 1ull : 0ull);
        tstart[m + 1] = tstart[m] + tiles[m];
    }
    const uint64_t U = ustart[M], T = tstart[M];
    // rounds of G pieces of min_piece tiles or more (one round at least)
    const uint64_t P = (uint64_t)G * std::max<uint64_t>(1ull, T / ((uint64_t)G * std::max(1u, min_piece)));
    std::vector<uint64_t> cut(P + 1);  // cut p (0..P) as a flattened tile coordinate
    uint32_t m = 0;
    for (uint64_t p = 0; p < P; ++p) {
        const uint64_t x = U * p / P;
        while (m < M && x >= ustart[m + 1]) ++m;
        const uint64_t off = m < M && x > ustart[m] ? x - ustart[m] - 1ull : 0ull;  // tiles of m before the cut
        cut[p] = m < M ? tstart[m] + std::min<uint64_t>(off, tiles[m]) : T;
    }
    cut[P] = T;
    std::vector<std::vector<Run>> piece_runs(P);
    std::vector<uint32_t> nruns(M, 0u);
    m = 0;
    for (uint64_t p = 0; p < P; ++p) {
        for (uint64_t g = cut[p]; g < cut[p + 1];) {
            while (g >= tstart[m + 1]) ++m;
            const uint64_t e = std::min(cut[p + 1], tstart[m + 1]);
            piece_runs[p].push_back(Run{m, (uint32_t)(g - tstart[m]), (uint32_t)(e - g), nruns[m]++, 0u, {0u, 0u, 0u}});
            g = e;
        }
    }
    runs.clear();
    block_runs.assign(G + 1, 0u);
    for (uint32_t b = 0; b < G; ++b) {
        block_runs[b] = (uint32_t)runs.size();
        for (uint64_t p = b; p < P; p += G)
            for (Run r : piece_runs[p]) {
                r.shares = nruns[r.seg];  // the member's parents prefetched in shares, one per run
                runs.push_back(r);
            }
    }
    block_runs[G] = (uint32_t)runs.size();
}

int build_group_launch(const std::vector<const PopView *> &members, uint32_t words, char *table, size_t table_capacity,
                       GenLaunch &gl, cudaStream_t stream) {
    if (members.empty()) {
        gl = GenLaunch{};
        return SPG_OK;
    }
    // records of 2L int16, words = L / 2: one block per 256 offspring
    OffspringKernel k = continuous_kernel(2u * words, members.size() > 1);
    int rc = prepare_offspring(k);
    if (rc != SPG_OK) return fail(rc, "offspring kernel setup failed");
    std::vector<Segment> segs;
    std::vector<uint32_t> bucket_map, tile_map;
    segs.reserve(members.size());
    uint32_t total_tiles = 0, buckets = 0;
    uint64_t offspring = 0;
    for (uint32_t si = 0; si < members.size(); ++si) {
        const PopView &v = *members[si];
        const uint32_t nt = (v.n + kBlock - 1) / kBlock;
        segs.push_back(segment_at(v.base, v.L, v.n, nt, total_tiles, v.nbuckets, buckets));
        tile_map.insert(tile_map.end(), nt, si);
        bucket_map.insert(bucket_map.end(), v.nbuckets, si);
        total_tiles += nt;
        buckets += v.nbuckets;
        offspring += v.n;
    }
    if (group_table_bytes((uint32_t)segs.size(), offspring, buckets) > table_capacity)
        return fail(SPG_ERR_INVALID, "launch table does not fit its buffer");
    const size_t off_buckets = align_up(segs.size() * sizeof(Segment), 256);
    const size_t off_tiles = off_buckets + align_up((size_t)buckets * 4, 256);
    cudaError_t e = cudaMemcpyAsync(table, segs.data(), segs.size() * sizeof(Segment), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(table + off_buckets, bucket_map.data(), bucket_map.size() * 4, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(table + off_tiles, tile_map.data(), tile_map.size() * 4, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);  // the host tables go away
    if (e != cudaSuccess) return cuda_fail(e, "upload launch table");
    gl = GenLaunch{};
    gl.offspring = k;
    gl.compact = compact_kernel();
    gl.args.segs = reinterpret_cast<const Segment *>(table);
    gl.args.bucket_seg = reinterpret_cast<const uint32_t *>(table + off_buckets);
    gl.args.tile_seg = reinterpret_cast<const uint32_t *>(table + off_tiles);
    gl.args.nsegs = (uint32_t)segs.size();
    if (segs.size() == 1) {
        gl.args.one = segs[0];
        gl.args.nsegs = 1;
    }
    gl.args.total_tiles = total_tiles;
    gl.args.total_buckets = buckets;
    gl.blocks = total_tiles;  // not persistent
    gl.buckets = buckets;
    return SPG_OK;
}

// ------------------------------------------------- one population's memory
int view_sync(const PopView &v) {
    const cudaError_t e = cudaStreamSynchronize(v.stream);
    return e == cudaSuccess ? SPG_OK : cuda_fail(e, "cudaStreamSynchronize");
}

// One copy in stream order: it waits for what the stream has to do, so no
// synchronisation goes before it.
static int read_back(const PopView &v, void *host, size_t off, size_t bytes, const char *what) {
    cudaError_t e = cudaMemcpyAsync(host, v.base + off, bytes, cudaMemcpyDeviceToHost, v.stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(v.stream);
    return e == cudaSuccess ? SPG_OK : cuda_fail(e, what);
}

int view_state(const PopView &v, DevState &st) { return read_back(v, &st, v.L.state, sizeof st, "read state"); }

int view_set_state(const PopView &v, uint32_t gen, uint32_t S, uint32_t f, double R, int32_t status,
                   uint32_t target) {
    return launch_set_state(reinterpret_cast<DevState *>(v.base + v.L.state),
                            reinterpret_cast<StatAcc *>(v.base + v.L.acc), gen, S, f, R, status, target, v.stream);
}

// The slot layout of generation `gen` of a single population from its full
// records and survivor list (null: everyone).
int view_pack(const PopView &v, uint32_t gen, const uint32_t *surv, uint32_t S) {
    const uint32_t par = gen & 1u;
    return launch_pack(reinterpret_cast<const PopParams *>(v.base + v.L.params), v.words,
                       reinterpret_cast<const uint32_t *>(v.base + v.L.geno0), surv, S, v.n, slot_length(v.n),
                       slot_count(v.n), reinterpret_cast<uint32_t *>(v.base + v.L.alive),
                       reinterpret_cast<uint32_t *>(v.base + v.L.packed[par]),
                       reinterpret_cast<uint32_t *>(v.base + v.L.counts[par]),
                       v.L.weighted ? reinterpret_cast<uint2 *>(v.base + v.L.mate[par]) : nullptr,
                       reinterpret_cast<GenAcc *>(v.base + v.L.gen_acc),
                       reinterpret_cast<unsigned long long *>(v.base + v.L.barrier), v.stream);
}

// Enqueue the generation-0 set-up of one population: parameters, counters,
// founders and state.  `prm` and `init_genotypes` must stay valid until the
// stream has run the copies (callers synchronise before returning).
int view_init(const PopView &v, const PopParams &prm, const uint32_t *init_genotypes, uint32_t p0_q32) {
    cudaError_t e = cudaSuccess;
    if (!v.L.solo) e = cudaMemsetAsync(v.base + v.L.buckets, 0, (size_t)2 * v.nbuckets * 4, v.stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(v.base + v.L.ring, 0, (size_t)v.cap * sizeof(spg_stats), v.stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(v.base + v.L.params, &prm, sizeof(PopParams), cudaMemcpyHostToDevice, v.stream);
    if (e != cudaSuccess) return cuda_fail(e, "initialise device memory");
    uint32_t *geno0 = reinterpret_cast<uint32_t *>(v.base + v.L.geno0);
    uint32_t *surv0 = reinterpret_cast<uint32_t *>(v.base + v.L.surv0);
    int rc;
    if (init_genotypes) {
        e = cudaMemcpyAsync(geno0, init_genotypes, (size_t)v.n * 2 * v.words * 4, cudaMemcpyHostToDevice, v.stream);
        if (e != cudaSuccess) return cuda_fail(e, "upload founders");
        rc = launch_iota(surv0, v.n, v.stream);
    } else if (prm.continuous) {
        rc = launch_founders_cont(reinterpret_cast<const PopParams *>(v.base + v.L.params), prm.n_loci, geno0, surv0,
                                  v.n, p0_q32, v.stream);
    } else {
        rc = launch_founders(v.words, geno0, surv0, v.n, prm.key0, prm.key1, prm.rep, p0_q32, v.stream);
    }
    if (rc != SPG_OK) return fail(rc, "founder launch failed");
    if (v.L.solo) {
        rc = view_pack(v, 0, nullptr, v.n);
        if (rc != SPG_OK) return fail(rc, "founder packing failed");
    }
    rc = view_set_state(v, 0, v.n, kCertain, 0.0, SPG_OK, 0xFFFFFFFFu);
    return rc == SPG_OK ? SPG_OK : fail(rc, "state launch failed");
}

int check_ecology(const spg_ecology *eco) {
    if (!eco) return fail(SPG_ERR_INVALID, "ecology is NULL");
    if (!eco->attack) return fail(SPG_ERR_INVALID, "attack table is NULL");
    if (!(eco->K > 0.0) || !(eco->R_half > 0.0) || !(eco->R0 >= 0.0) || !std::isfinite(eco->r) ||
        !std::isfinite(eco->K) || !std::isfinite(eco->R0))
        return fail(SPG_ERR_INVALID, "ecology needs K > 0, R_half > 0, R0 >= 0, finite r");
    if (eco->model > 1u) return fail(SPG_ERR_INVALID, "ecology model must be 0 (logistic) or 1 (Beverton-Holt)");
    if (!(eco->r_sd >= 0.0) || !std::isfinite(eco->r_sd) || (eco->model == 0u && eco->r_sd != 0.0))
        return fail(SPG_ERR_INVALID, "r_sd must be finite, >= 0, and 0 for the logistic resource");
    return SPG_OK;
}

// Attach an ecology: parameters (host copy updated and uploaded, then the
// stream synchronised) and the state's R and f.
int view_set_ecology(const PopView &v, PopParams &prm, const spg_ecology *eco) {
    int rc = check_ecology(eco);
    if (rc != SPG_OK) return rc;
    DevState st;
    rc = view_state(v, st);
    if (rc != SPG_OK) return rc;
    std::memcpy(prm.attack, eco->attack, sizeof prm.attack);
    prm.has_eco = 1;
    prm.eco_model = eco->model;
    prm.r_sd = eco->r_sd;
    prm.r = eco->r;
    prm.K = eco->K;
    prm.R_half = eco->R_half;
    const cudaError_t e =
        cudaMemcpyAsync(v.base + v.L.params, &prm, sizeof(PopParams), cudaMemcpyHostToDevice, v.stream);
    if (e != cudaSuccess) return cuda_fail(e, "upload parameters");
    rc = view_set_state(v, st.gen, st.S, factor_q32_host(eco->R0, eco->R_half), eco->R0, st.status, st.target);
    if (rc != SPG_OK) return rc;
    return view_sync(v);
}

// Bytes of state and ring that one copy brings at the price of a copy of the
// state alone.
constexpr size_t kReadTogether = 48u << 10;

int view_read_stats(const PopView &v, uint32_t first_gen, uint32_t count, spg_stats *out) {
    if (!out && count) return fail(SPG_ERR_INVALID, "NULL argument");
    // the state and, when the ring is short, the ring behind it in one copy
    // (two copies when the host has no memory for that)
    DevState st;
    const size_t ring_at = v.L.ring - v.L.state, all = ring_at + (size_t)v.cap * sizeof(spg_stats);
    const std::unique_ptr<char[]> both(all <= kReadTogether ? new (std::nothrow) char[all] : nullptr);
    int rc;
    if (both) {
        rc = read_back(v, both.get(), v.L.state, all, "read state and stats");
        if (rc == SPG_OK) std::memcpy(&st, both.get(), sizeof st);
    } else {
        rc = view_state(v, st);
    }
    if (rc != SPG_OK) return rc;
    if (count == 0) return SPG_OK;
    const uint64_t last = (uint64_t)first_gen + count - 1;
    if (first_gen == 0 || last > st.gen || (uint64_t)st.gen - first_gen >= v.cap)
        return fail(SPG_ERR_RANGE, "generations %u..%llu not in the ring (completed %u, capacity %u)", first_gen,
                    (unsigned long long)last, st.gen, v.cap);
    const spg_stats *ring = reinterpret_cast<const spg_stats *>(v.base + v.L.ring);
    for (uint32_t i = 0; i < count;) {
        const uint32_t slot = (first_gen - 1 + i) % v.cap;
        const uint32_t run = std::min(count - i, v.cap - slot);
        if (both) {
            std::memcpy(out + i, both.get() + ring_at + slot * sizeof(spg_stats), run * sizeof(spg_stats));
        } else {
            const cudaError_t e = cudaMemcpy(out + i, ring + slot, run * sizeof(spg_stats), cudaMemcpyDeviceToHost);
            if (e != cudaSuccess) return cuda_fail(e, "read stats");
        }
        i += run;
    }
    return st.status < 0 ? fail(st.status, "device status %d", st.status) : SPG_OK;
}

// Rows of per-locus counts of generations first_gen .. first_gen+count-1
// from a population's ring: counted generations are from .. min(until, the
// current one) and the ring keeps the last la.cap of them.
int read_locus_rows(const LocusArgs &la, uint32_t n_loci, uint32_t from, uint32_t until, const DevState &st,
                    uint32_t first_gen, uint32_t count, uint32_t *out) {
    if (count == 0) return SPG_OK;
    const uint64_t last = (uint64_t)first_gen + count - 1;
    until = std::min(until, st.gen);
    if (first_gen == 0 || first_gen < from || last > until || (uint64_t)st.gen - first_gen >= la.cap)
        return fail(SPG_ERR_RANGE, "per-locus counts of generations %u..%llu not kept (counted %u..%u, capacity %u)",
                    first_gen, (unsigned long long)last, from, until, la.cap);
    const size_t row = n_loci;
    for (uint32_t i = 0; i < count;) {
        const uint32_t slot = (first_gen - 1 + i) % la.cap;
        const uint32_t run = std::min(count - i, la.cap - slot);
        const cudaError_t e = cudaMemcpy(out + (size_t)i * row, la.ring + (size_t)slot * row, run * row * 4u,
                                         cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return cuda_fail(e, "read per-locus counts");
        i += run;
    }
    return st.status < 0 ? fail(st.status, "device status %d", st.status) : SPG_OK;
}

int view_read_genotypes(const PopView &v, uint32_t *host, size_t n_words) {
    if (!host) return fail(SPG_ERR_INVALID, "NULL argument");
    const size_t need = (size_t)v.n * 2 * v.words;
    if (n_words < need) return fail(SPG_ERR_INVALID, "buffer holds %zu words, need %zu", n_words, need);
    DevState st;
    int rc = view_state(v, st);
    if (rc != SPG_OK) return rc;
    const char *src = v.base + ((st.gen & 1u) ? v.L.geno1 : v.L.geno0);
    const cudaError_t e = cudaMemcpy(host, src, need * 4, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? SPG_OK : cuda_fail(e, "read genotypes");
}

int view_read_survivors(const PopView &v, uint32_t *host, size_t capacity, uint32_t *S) {
    if (!S) return fail(SPG_ERR_INVALID, "NULL argument");
    DevState st;
    int rc = view_state(v, st);
    if (rc != SPG_OK) return rc;
    *S = st.S;
    if (!host) return SPG_OK;
    if (capacity < st.S) return fail(SPG_ERR_INVALID, "buffer holds %zu, need %u", capacity, st.S);
    const char *src = v.base + ((st.gen & 1u) ? v.L.surv1 : v.L.surv0);
    const cudaError_t e = cudaMemcpy(host, src, (size_t)st.S * 4, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? SPG_OK : cuda_fail(e, "read survivors");
}

int view_get_state(const PopView &v, spg_state *out) {
    if (!out) return fail(SPG_ERR_INVALID, "NULL argument");
    DevState st;
    const int rc = view_state(v, st);
    if (rc != SPG_OK) return rc;
    out->gen = st.gen;
    out->S = st.S;
    out->status = st.status;
    out->f = st.f;
    out->R = st.R;
    return SPG_OK;
}

}  // namespace spg


using namespace spg;

extern "C" {
uint32_t spg_abi_version(void) { return SPG_ABI_VERSION; }

uint32_t spg_mutation_cdf(double mu, uint32_t n_copies, uint32_t cdf[32]) {
    if (!cdf || !(mu >= 0.0 && mu < 1.0)) return 0;
    return mutation_cdf(mu, n_copies, cdf);
}

const char *spg_last_error(void) { return g_last_error.c_str(); }

const char *spg_status_string(int code) {
    switch (code) {
        case SPG_OK: return "ok";
        case SPG_EXTINCT: return "extinct: no survivors";
        case SPG_ERR_INVALID: return "invalid argument";
        case SPG_ERR_OOM: return "device allocation failed";
        case SPG_ERR_CUDA: return "CUDA runtime error";
        case SPG_ERR_TIMEOUT: return "bounded device wait timed out";
        case SPG_ERR_RANGE: return "generations not available";
        case SPG_ERR_BUDGET: return "memory budget exceeded";
        default: return "unknown status";
    }
}

void spg_summarize(const spg_stats *st, uint32_t n_loci, float out[5]) {
    const double n = (double)st->n;
    const double mean_raw = (double)st->sum_raw / n;
    const double second = (double)st->sum_raw2 / n;
    const double sq = mean_raw * mean_raw;
    const double var_raw = second - sq;
    out[0] = (float)(mean_raw / 512.0);
    out[1] = (float)(var_raw / (512.0 * 512.0));
    out[2] = (float)((double)st->s / n);
    out[3] = (float)((double)st->het / (n * (double)n_loci));
    out[4] = (float)((double)st->allele / (2.0 * n * (double)n_loci));
}

}  // extern "C"
