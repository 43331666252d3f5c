// Internal types shared by the host engine and the kernels of libspegg_gb300.
// Not part of the C ABI (include/spegg.h is).
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "spegg.h"

namespace spg {

constexpr int kBins = 4096;
constexpr int kMaxKmax = 32;      // entries of the Binomial(2L, mu) CDF table
constexpr int kMutDraws = 64;     // position draws tried per offspring
constexpr int kMaxPlanes = 16;    // bit planes of the offset-binary effects
constexpr int kMaxWords = 8;      // W = L/32 <= 8
constexpr int kBlock = 256;       // threads per block of the continuous-allele kernel
constexpr int kLutWords = 256;    // entries of one byte table (one per byte value)
constexpr uint32_t kBucket = 4096;                 // offspring per compaction bucket
constexpr uint32_t kBucketWords = kBucket / 32;    // bitmap words per bucket = compaction threads
constexpr uint32_t kCompactCopyThreads = 256;  // threads that write a bucket's survivors (8 warps)
constexpr uint32_t kCompactThreads = kCompactCopyThreads + 32;  // + one warp that closes the generation
constexpr uint32_t kCertain = 0xFFFFFFFFu;
constexpr int kAccCopies = 16;    // copies of the statistics accumulators (spread atomics)

constexpr int kMaxLoci = 256;
constexpr int kMaxLutBytes = kMaxLoci / 8;  // byte positions of a haplotype (L / 8)
constexpr int kMaxChrom = 96;            // chromosomes of a linkage map
constexpr uint32_t kLinkSites = 65536;   // crossover opportunities per gamete
constexpr double kMaxMapMorgans = 16.0;  // total length of a linkage map
constexpr int kLinkGuideBits = 12;       // the crossover uniform's top bits that index the guide table
constexpr int kLinkGuide = 1 << kLinkGuideBits;

// Philox counter word 3 = purpose << 24 | sub
enum Purpose : uint32_t {
    kFounder = 1, kMate = 2, kRecomb = 3, kMutPos = 4, kLink = 5, kMateW = 6, kGrowth = 7, kMutSize = 8, kEnv = 9
};
constexpr uint32_t kMateAttempts = 64;   // proposals per weighted parent

// Acceptance thresholds of weighted parents (device global memory): acc[0]
// mothers, acc[1] fathers, by phenotype bin (Q32, 0xFFFFFFFF = always).
struct alignas(16) WeightParams {
    uint32_t acc[2][kBins];
};

// Tables of a linkage map (device global memory, one per linked population).
struct alignas(16) LinkParams {
    uint32_t cdf[kMaxKmax];      // crossover count per gamete, Binomial(kLinkSites, D / kLinkSites) CDF, Q32
    uint32_t cum[kMaxLoci];      // interval CDF, Q32: crossover interval = #{l <= L-2 : cum[l] <= u}
    // bucket h of crossover uniforms (u >> 20 == h): interval I0 of u = h << 20
    // (bits 0-7), and how many cum[l] (l <= L-2) lie inside the bucket (bits
    // 26-27: 0, 1, or 2 = two or more)
    uint32_t guide[kLinkGuide];
    uint16_t first[kMaxChrom];   // first locus of each chromosome
    uint32_t kmax;               // entries of cdf
    uint32_t nchrom;
};

// Read-only parameters of one population (device global memory).
struct alignas(16) PopParams {
    uint32_t table[kBins];                  // viability thresholds per bin
    uint32_t attack[kBins];                 // Q16 attack rate per bin (ecology)
    uint32_t planes[kMaxPlanes * kMaxWords];// plane b, word w at [b * W + w]
    uint32_t dplanes[kMaxPlanes * kMaxWords];// dominance deviations, offset binary like planes
    int32_t d_min;                          // dominance = d_min + sum_b 2^b * dplane_b
    uint32_t ndplanes;                      // 0: additive genetic value
    uint32_t has_dom;                       // some locus has a non-zero dominance deviation
    // byte tables of the genetic value: lut[k * 256 + v] is the sum of the
    // effects of loci 8k .. 8k+7 whose bit is set in v (L / 8 tables; the
    // allocation-free call)
    alignas(16) int32_t lut[kMaxLutBytes * kLutWords];
    uint32_t cdf[kMaxKmax];                 // Binomial(2L, mu) CDF, Q32
    int32_t e_min;                          // effects = e_min + sum_b 2^b * plane_b
    uint32_t nplanes;
    int32_t bias;
    uint32_t shift;
    uint32_t kmax;
    uint32_t n;
    uint32_t n_loci;
    uint32_t words;
    uint32_t key0, key1, rep;
    uint32_t has_eco;
    double r, K, R_half;
    double r_sd;                 // Beverton-Holt: sd of the growth rate
    uint32_t eco_model;          // 0 logistic, 1 Beverton-Holt
    uint32_t continuous;         // allelic values are int16 Q8 (records of L words)
    long long s_mut, s_env;      // continuous: Irwin-Hall step scales, Q16
    uint32_t ntiles;
    uint32_t stats_cap;
    const LinkParams *link;      // linkage map tables, or null (free recombination)
    uint32_t linked;
    uint32_t weighted;           // parents drawn by weight (weights != null)
    const WeightParams *weights;
};

// the generation kernel and the allocation-free call's offspring kernel copy
// these tables with 16-byte cp.async
static_assert(offsetof(PopParams, table) % 16 == 0 && offsetof(PopParams, attack) % 16 == 0 &&
                  offsetof(PopParams, lut) % 16 == 0,
              "tables copied in 16-byte chunks");

// Mutable per-population state (device global memory).
struct alignas(16) DevState {
    uint32_t gen;     // generations completed
    uint32_t S;       // survivors of generation `gen` (parents of the next)
    uint32_t f;       // resource factor applied to the next generation
    int32_t status;   // SPG_OK or SPG_EXTINCT
    double R;         // resource density
    uint32_t done;    // compaction buckets of the running generation that have finished;
                      // biallelic: the generation that k_close has to close, or 0
    uint32_t target;  // generations stop once gen reaches target (0xFFFFFFFF: never)
    // the generation being closed: computed while its survivors are being
    // compacted, committed by the block that finishes the last bucket
    uint32_t next_S, next_f;
    int32_t next_status;
    uint32_t pad;
    double next_R;
};

// Statistics of the generation being formed, accumulated by atomics; each
// population has kAccCopies copies on separate cache lines.
struct alignas(128) StatAcc {
    unsigned long long s;
    long long sum_raw, sum_raw_s;
    unsigned long long sum_raw2, cons, het, allele;
    int mn, mx;
};

// One population as seen by a generation launch.
struct alignas(16) Segment {
    const PopParams *prm;
    uint32_t *geno[2];                // ping-pong genotype buffers [N * 2W]
    uint32_t *surv[2];                // ping-pong survivor lists [N]
    uint32_t *alive;                  // alive bitmap of the generation being formed [nbuckets * kBucketWords]
    uint32_t *bucket_sum;             // survivors per bucket, by generation parity [2][nbuckets]
    DevState *state;
    StatAcc *acc;                     // [kAccCopies]
    spg_stats *ring;                  // [stats_cap]
    uint32_t n;                       // offspring per generation
    uint32_t tile_begin;              // first launch-wide tile of this population
    uint32_t ntiles;
    uint32_t bucket_begin;            // first launch-wide bucket of this population
    uint32_t nbuckets;
    uint32_t pad;
};

// A run of a block of a launch group (schedule_runs): tiles tile0 .. tile0 +
// count - 1 of member seg, whose tiles are split into `shares` runs (this is
// run `share`).
struct alignas(16) Run {
    uint32_t seg, tile0, count, share, shares, pad[3];
};

struct GenArgs {
    const Segment *segs;         // device array of nsegs segments (used when nsegs > 1)
    const uint32_t *bucket_seg;  // segment of each launch-wide bucket (nsegs > 1)
    const uint32_t *tile_seg;    // segment of each launch-wide tile (nsegs > 1)
    uint32_t nsegs;
    uint32_t total_tiles;        // tiles of the single segment (nsegs == 1: contiguous shares per block)
    uint32_t total_buckets;
    Segment one;           // the segment itself when nsegs == 1 (read from kernel parameters)
};

using GenKernel = void (*)(GenArgs);

// A single population's generations (generations.cuh).  Its groups of 32
// offspring are cut into slots of slot_len groups; a generation's survivors
// are packed slot by slot in packed[generation & 1], counts[generation & 1]
// holding their number per slot.
constexpr uint32_t kSoloThreads = 512;  // (768 and 1,024 threads spill: 1.1 and 1.4 times the time at L = 32)
constexpr uint32_t kMaxSlots = 152 * (kSoloThreads / 32);  // one per resident warp on 152 SMs
constexpr uint32_t kOneBlockGroups = 16;  // groups up to which one block is no slower than several and a grid barrier
// The per-locus values as f16 elements, laid out as the matrix fragments of
// the generation kernel (value_fragments): the additive values, or with
// dominance those of heterozygous and of homozygous loci.
struct alignas(16) ValueFragments {
    uint32_t table[2][1024];
};
// Statistics of the generation being formed, in kGenAccCopies copies (block b
// adds to copy b % kGenAccCopies); three generations' worth, by generation % 3.
struct alignas(64) GenAcc {
    unsigned long long sum[6];  // raw, raw over survivors, raw^2, consumption, heterozygosity, alleles
    int mn, mx;
    unsigned long long pad;
};
constexpr uint32_t kGenAccCopies = 4;
constexpr unsigned long long kEmptyMinMax = 0x800000007FFFFFFFull;  // mx INT_MIN over mn INT_MAX
constexpr uint32_t kBarrierTries = 1u << 24;  // polls of about half a microsecond before a wait gives up
constexpr int kMaxGuideBits = 13;  // the parent draw's top bits that index the directory's guide, at most
struct alignas(16) SoloArgs {
    uint32_t keys[20];                 // Philox round keys (word 0, word 1 of each round)
    const PopParams *prm;
    const ValueFragments *frag;
    uint32_t *packed[2];               // survivors' records by generation parity [N * 2W]
    uint2 *mate[2];                    // weighted parents: their thresholds as mother and father, same places
    uint32_t *counts[2];               // survivors per slot [nslots]
    uint32_t *geno;                    // full records of the last generation of a call [N * 2W]
    uint32_t *alive;                   // its survivor bitmap
    uint32_t *surv;                    // its ordered survivor list [N]
    DevState *state;
    GenAcc *acc;                       // [3][kGenAccCopies], by generation % 3
    unsigned long long *barrier;       // grid barrier arrivals (generations.cuh)
    spg_stats *ring;
    uint32_t *locus_row[2];            // per-locus counts of the generation being formed, by parity (null: off)
    uint32_t *locus_ring;              // [locus_cap][L]
    uint32_t locus_cap;
    uint32_t n, slot_len, nslots, guide_bits;
    uint32_t words;                    // W = L / 32
    uint32_t rep, kmax, shift;
    uint32_t mut_from;                 // mutation draws from here on count a mutation (kmax 0: none do)
    int32_t bias;
    uint32_t narrow_bias;              // genetic value + bias fits 32 bits
    uint32_t has_eco, eco_model, stats_cap;
    double eco_r, eco_r_sd, eco_K, eco_R_half;
    uint32_t dom, two_digits;          // fragments: dominance, values beyond 2048 in magnitude
    uint32_t n_gen;                    // generations of this launch
    uint32_t keep_last;                // the last of them is the call's last
    uint32_t single;                   // one generation without a grid barrier: k_close closes it
    uint32_t barrier_tries;            // polls of a wait before it gives up
    uint32_t close_slots;              // slots whose survivors a block of k_close lists, at most 256
};
struct SoloKernel {
    const void *fn = nullptr;
    uint32_t smem = 0, resident = 0;  // resident: blocks on the device at a time
};
SoloKernel solo_kernel(uint32_t words, bool linked, bool weighted, bool general);
const void *close_kernel();          // k_close
const void *close_members_kernel();  // k_close_members
int prepare_close();         // sets its shared-memory limit
constexpr uint32_t kCloseThreads = 256 + 32;  // + one warp that closes the generation
constexpr uint32_t kCloseSmem = 120000;  // not used: keeps its blocks on an SM each
int prepare_solo(SoloKernel &k);  // sets the shared-memory limit, fills `resident`

// Several populations in one launch (k_teams): block b works through places
// block_places[b] .. block_places[b + 1] - 1, being block `rank` of `team` for
// population `member`.
struct TeamPlace {
    uint32_t member;
    uint16_t rank, team;
};
struct TeamArgs {
    const SoloArgs *members;
    const TeamPlace *places;
    const uint32_t *block_places;
    uint32_t n_gen, keep_last;
    uint32_t single;  // one generation without barriers: k_close_members closes it
};
// Block b of k_close_members closes slots from part * close_slots of a member.
struct ClosePart {
    const SoloArgs *member;
    uint32_t part, pad;
};
// Kinds of members that share a launch: plain ones, general values, linkage
// map, parent weights, both.
constexpr uint32_t kTeamKinds = 5;
inline uint32_t team_kind(bool linked, bool weighted, bool general) {
    return linked ? (weighted ? 4u : 2u) : weighted ? 3u : general ? 1u : 0u;
}
SoloKernel team_kernel(uint32_t kind);
// Enqueue the slot layout of a generation: bitmap words and per-slot counts
// of the survivors (surv: their ordered list of S, null for all n), their
// records packed[slot ...] and, when mate is given, their parent thresholds;
// the accumulators and the barrier counter start empty.
int launch_pack(const PopParams *prm, uint32_t words, const uint32_t *geno, const uint32_t *surv, uint32_t S, uint32_t n,
                uint32_t slot_len, uint32_t nslots, uint32_t *alive, uint32_t *packed, uint32_t *counts, uint2 *mate,
                GenAcc *acc, unsigned long long *barrier, void *stream);

// Launch shape of a population or a batch's locus count, as callers set and
// read it: threads per block, offspring per thread (per lane pair when lanes
// = 2) and lanes per offspring (1, or 2 for L >= 128).  Results never depend
// on it, and the generation kernel has one shape of its own.
struct Shape {
    uint32_t block = 256, items = 1, lanes = 1;
};
bool supported_shape(uint32_t words, const Shape &shape);

// The kernel that forms a generation's offspring where a compaction follows
// it (256 threads): entry, offspring per tile, dynamic shared memory, blocks
// resident on the device, and whether it may start while its predecessor
// finishes.  The allocation-free call's (offspring.cu) is persistent; the
// continuous-allele one (kernels.cu) runs one block per tile.
struct OffspringKernel {
    GenKernel fn = nullptr;
    uint32_t tile = 0, smem = 0, resident = 0;
    bool programmatic = false;
};
OffspringKernel offspring_kernel(uint32_t words);
int prepare_offspring(OffspringKernel &k);  // sets the shared-memory limit, fills `resident`
GenKernel compact_kernel();                 // the compaction kernel

constexpr int kLocusPlanes = 5;  // bit-sliced counter planes per lane (31 records between flushes)
// Per-locus allele counts of a population (optional, biallelic records): the
// counts of the generations kept in a ring [cap][L] (generation g in slot
// (g - 1) % cap) and the rows of the generations being formed [2][L], by
// parity.
struct LocusArgs {
    uint32_t *ring, *acc;
    uint32_t cap;
};
// Enqueue founders: generation-0 records by Philox draws, survivors = 0..n-1.
int launch_founders(uint32_t words, uint32_t *geno, uint32_t *surv, uint32_t n, uint32_t key0, uint32_t key1,
                    uint32_t rep, uint32_t p0_q32, void *stream);
// Enqueue survivors = 0..n-1 only (caller-supplied founders).
int launch_iota(uint32_t *surv, uint32_t n, void *stream);
// The generation kernel of a continuous-allele population (one warp per
// offspring at a time, 256 offspring per block, no persistent grid).
OffspringKernel continuous_kernel(uint32_t n_loci, bool group = false);  // group: several populations (tile map)
// Enqueue continuous founders: value = effect[l] * allele of the biallelic
// founder draws (records of 2L int16), survivors = 0..n-1.
int launch_founders_cont(const PopParams *prm, uint32_t n_loci, uint32_t *geno, uint32_t *surv, uint32_t n,
                         uint32_t p0_q32, void *stream);
// Enqueue a state reset: state fields and cleared statistics accumulators.
int launch_set_state(DevState *st, StatAcc *acc, uint32_t gen, uint32_t S, uint32_t f, double R, int32_t status,
                     uint32_t target, void *stream);

}  // namespace spg
