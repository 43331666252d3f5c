// Host-side helpers shared by the population, batch and server engines.
#pragma once

#include <cuda_runtime.h>

#include <cstdarg>
#include <cstddef>
#include <cstdint>
#include <vector>

#include "spegg.h"
#include "spegg_internal.h"

namespace spg {

constexpr uint32_t kGraphChunk = 32;          // generations per cached graph
constexpr uint32_t kCheckpointMagic = 0x43475053u;  // "SPGC"

struct CheckpointHeader {
    uint32_t magic, version, n, n_loci, gen, S;
    int32_t status;
    uint32_t f;
    double R;
    uint64_t seed;
    uint32_t replicate, pad;
};

struct Allocator {
    spg_allocator hooks{nullptr, nullptr, nullptr};
    void *alloc(size_t bytes, cudaStream_t s) const;
    void release(void *p, cudaStream_t s) const;
};

// Byte offsets of one population's buffers inside its arena.
struct PopLayout {
    size_t params, state, acc, geno0, geno1, surv0, surv1, alive, buckets, ring, segment, link;
    size_t weights;  // weighted parents only (0 otherwise)
    bool weighted;
    // a single biallelic population (solo_layout_for): geno0 = geno1 and
    // surv0 = surv1, no buckets or segment
    bool solo;
    size_t packed[2], counts[2], mate[2], gen_acc, barrier, frag;
    size_t total;
};

// One population's device memory: its arena, layout and sizes.
struct PopView {
    char *base = nullptr;
    PopLayout L{};
    uint32_t n = 0, words = 0, cap = 0, nbuckets = 0;
    cudaStream_t stream = nullptr;
};

// The two launches of one generation for a launch group.
struct GenLaunch {
    OffspringKernel offspring;
    GenKernel compact = nullptr;
    GenArgs args{};
    uint32_t blocks = 0;   // offspring grid: min(tiles, resident blocks)
    uint32_t buckets = 0;  // compaction grid
};

// A cached CUDA graph of `length` generations (2 dependent launches each).
struct GraphChain {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    uint32_t length = 0;
    ~GraphChain();
    void reset();
    int build(const GenLaunch &gl, uint32_t len);
};

// Generations of several biallelic populations in shared launches (k_teams).
constexpr uint32_t kSoloLaunchGens = 512;  // generations of one launch of the generation kernel, at most
struct TeamMember {
    const SoloArgs *args = nullptr;  // (read when the tables are built)
    uint32_t n = 0, words = 0;
    bool linked = false, weighted = false, general = false;  // (the kind: team_kind)
};
struct TeamLaunch {
    std::vector<TeamMember> members;  // of one kind
    SoloKernel kernel;
    TeamArgs args{};
    char *table = nullptr;            // the members' arguments and the blocks' places
    size_t capacity = 0;
    uint32_t blocks = 0;              // of its launches
    double cycles = 0.0;              // estimated cycles of a generation of all members
    cudaStream_t side = nullptr;      // its launches' stream, beside the other kinds'
    cudaEvent_t joined = nullptr;
    void release(const Allocator &alloc, cudaStream_t stream);
};
struct TeamSet {
    TeamLaunch launch[kTeamKinds];
    bool beside = false;              // the kinds' launches run side by side
    cudaEvent_t forked = nullptr;
    ClosePart *parts = nullptr;       // calls of one generation: k_close_members' blocks
    uint32_t nparts = 0;
    size_t parts_capacity = 0;
    // singles: calls of one generation are formed without barriers; `kept`: work of
    // other launches that run beside these, in SM cycles a generation, and the most
    // SMs it fills (0: none).  Synchronises.
    int build(const std::vector<TeamMember> &all, const Allocator &alloc, cudaStream_t stream, bool singles,
              double kept = 0.0, uint32_t kept_blocks = 0);
    int update(const SoloArgs *args, cudaStream_t stream);
    int step(uint32_t n_gen, bool keep_last, cudaStream_t stream);
    void release(const Allocator &alloc, cudaStream_t stream);
};
TeamMember team_member(const SoloArgs &a, bool linked, bool weighted);
uint32_t launch_generations(const TeamMember &m, uint32_t blocks, uint32_t resident);
double continuous_work(uint32_t n, uint32_t n_loci);
uint32_t continuous_blocks(uint32_t n);
std::vector<uint32_t> deal_blocks(const std::vector<double> &work, const std::vector<uint32_t> &most, uint32_t blocks);
double schedule_teams(const std::vector<TeamMember> &members, uint32_t blocks, std::vector<TeamPlace> &places,
                      std::vector<uint32_t> &block_places);
uint32_t most_blocks(uint32_t n, uint32_t resident);
uint32_t solo_grid(uint32_t n, uint32_t words, uint32_t resident);
void solo_args(const PopView &v, const PopParams &prm, SoloArgs &a);

int fail(int code, const char *fmt, ...);
int cuda_fail(cudaError_t e, const char *what);
uint32_t mutation_cdf(double mu, uint32_t n_copies, uint32_t *cdf);
void effect_planes(const int16_t *effects, uint32_t n_loci, PopParams &prm);
void byte_tables(const int16_t *v, uint32_t n_loci, int32_t *lut);
uint32_t factor_q32_host(double R, double R_half);
size_t align_up(size_t x, size_t a);
// Value fragments of the effects and dominance deviations (null: none);
// two_digits: some value is beyond 2048 in magnitude.
void value_fragments(const int16_t *effects, const int16_t *dominance, uint32_t n_loci, ValueFragments &vf,
                     uint32_t &two_digits);
int validate_desc(const spg_pop_desc *d);
int build_params(const spg_pop_desc *d, PopParams &prm);
// Linkage-map tables from map_morgans[L] (validated; see spegg.h).
int build_link(const double *map_morgans, uint32_t n_loci, LinkParams &lp);
// Acceptance thresholds from the mother and father weight tables (NULL: uniform).
int build_weights(const uint32_t *mother_w, const uint32_t *father_w, WeightParams &wp);
PopLayout layout_for(uint32_t n, uint32_t words, uint32_t nbuckets, uint32_t cap);
Segment segment_at(char *base, const PopLayout &L, uint32_t n, uint32_t ntiles, uint32_t tile_begin,
                   uint32_t nbuckets, uint32_t bucket_begin);
uint32_t bucket_count(uint32_t n);
uint32_t slot_length(uint32_t n);
uint32_t slot_count(uint32_t n);
PopLayout solo_layout_for(uint32_t n, uint32_t words, uint32_t cap, bool weighted);
int view_pack(const PopView &v, uint32_t gen, const uint32_t *surv, uint32_t S);
Shape default_shape(uint32_t words);
constexpr uint32_t kAutotuneCandidates = SPG_AUTOTUNE_CANDIDATES;  // launch shapes timed per group
Shape autotune_candidate(uint32_t words, uint32_t c);
int shape_from_abi(uint32_t words, const spg_launch_shape *in, Shape &out);
// One generation's launches (each kernel may start while its predecessor in
// the stream finishes; see griddep_wait in the kernels).
int launch_generation(const GenLaunch &gl, cudaStream_t stream);
// Append a chain of `len` generations of one launch group to a graph
// (kernel nodes joined by programmatic edges); params: the GenArgs pointer.
int add_generation_nodes(cudaGraph_t graph, const GenLaunch &gl, void **params, uint32_t len);
size_t group_table_bytes(uint32_t members, uint64_t offspring, uint32_t buckets);
int read_locus_rows(const LocusArgs &la, uint32_t n_loci, uint32_t from, uint32_t until, const DevState &st,
                    uint32_t first_gen, uint32_t count, uint32_t *out);
void schedule_runs(const std::vector<uint32_t> &tiles, uint32_t G, uint32_t min_piece, std::vector<Run> &runs,
                   std::vector<uint32_t> &block_runs);
// Segment table, tile and bucket maps of one group of continuous-allele
// members (words = L / 2, the int16 records' words), uploaded into `table`
// (device memory; synchronous), and the group's launch description.
int build_group_launch(const std::vector<const PopView *> &members, uint32_t words, char *table, size_t table_capacity,
                       GenLaunch &gl, cudaStream_t stream);
int view_sync(const PopView &v);
int view_state(const PopView &v, DevState &st);
int view_set_state(const PopView &v, uint32_t gen, uint32_t S, uint32_t f, double R, int32_t status,
                   uint32_t target);
int view_init(const PopView &v, const PopParams &prm, const uint32_t *init_genotypes, uint32_t p0_q32);
int check_ecology(const spg_ecology *eco);
int view_set_ecology(const PopView &v, PopParams &prm, const spg_ecology *eco);
int view_read_stats(const PopView &v, uint32_t first_gen, uint32_t count, spg_stats *out);
int view_read_genotypes(const PopView &v, uint32_t *host, size_t n_words);
int view_read_survivors(const PopView &v, uint32_t *host, size_t capacity, uint32_t *S);
int view_get_state(const PopView &v, spg_state *out);
int enqueue_generations(const GenLaunch &gl, uint32_t n_gen, GraphChain &chain, cudaStream_t stream);

}  // namespace spg
