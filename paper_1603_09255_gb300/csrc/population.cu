// C ABI of one population (spg_pop): create, ecology, stepping, reads,
// checkpoint/restore, tiling (see include/spegg.h).
//
// A population owns one device arena (parameters, state, statistics ring,
// accumulators, genotypes, survivors).  The generations of a biallelic
// population are formed by cooperative launches of many (launch_generations; a
// call of one generation takes two plain ones); those of continuous allelic
// values are enqueued as a cached CUDA graph of kGraphChunk generations (two
// launches each), whose arguments are identical because buffers are chosen on
// the device by generation parity.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <new>

#include "spegg.h"
#include "spegg_engine.h"
#include "spegg_internal.h"

using namespace spg;

struct spg_pop {
    uint32_t n = 0, n_loci = 0, words = 0, ntiles = 0, nbuckets = 0, cap = 0;
    Shape shape;
    uint64_t seed = 0;
    uint32_t rep = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    Allocator alloc;
    char *arena = nullptr;
    PopLayout L{};
    PopParams *host_prm = nullptr;  // host copy of the parameters
    ValueFragments frag{};          // fragments of the genetic value (biallelic records)
    LinkParams link{};              // linkage-map tables (when host_prm->linked)
    WeightParams *weights = nullptr;  // parent acceptance thresholds (when host_prm->weighted)
    SoloKernel solo;   // biallelic records: the generation kernel, its grid and arguments
    SoloArgs sa{};
    uint32_t solo_blocks = 0, launch_gens = 0;
    GenLaunch gl;      // continuous allelic values: generation and compaction launches
    GraphChain chain;
    // per-locus allele counts (off until spg_set_locus_counts): ring, partial
    // rows and counter in one allocation; readable from generation locus_from
    char *locus_mem = nullptr;
    LocusArgs locus{};
    bool locus_on = false;
    uint32_t locus_from = 0, locus_until = 0;  // counted generations: locus_from .. (on ? now : locus_until)

    PopView view() const {
        PopView v;
        v.base = arena;
        v.L = L;
        v.n = n;
        v.words = words;
        v.cap = cap;
        v.nbuckets = nbuckets;
        v.stream = stream;
        return v;
    }
};

namespace {

// The rows the generation kernel adds its per-locus counts to, or none.
void attach_locus(spg_pop *p) {
    for (uint32_t i = 0; i < 2; ++i) p->sa.locus_row[i] = p->locus_on ? p->locus.acc + (size_t)i * p->n_loci : nullptr;
    p->sa.locus_ring = p->locus.ring;
    p->sa.locus_cap = p->locus.cap;
}

// The generation kernel, its grid and its arguments.  The launch shape is
// accepted and reported; the kernel has one shape of its own (results never
// depend on it).
int configure_solo(spg_pop *p, const Shape &shape) {
    const PopParams &prm = *p->host_prm;
    SoloArgs &a = p->sa;
    solo_args(p->view(), prm, a);
    SoloKernel k = solo_kernel(p->words, prm.linked != 0u, prm.weighted != 0u, a.dom || a.two_digits || !a.narrow_bias);
    int rc = prepare_solo(k);
    if (rc == SPG_OK) rc = prepare_close();
    if (rc != SPG_OK) return fail(rc, "generation kernel setup failed");
    p->solo = k;
    p->shape = shape;
    p->solo_blocks = solo_grid(p->n, p->words, k.resident);
    p->launch_gens = launch_generations(team_member(a, prm.linked != 0u, prm.weighted != 0u), p->solo_blocks, k.resident);
    attach_locus(p);
    return SPG_OK;
}

// Blocks of a launch that forms one generation for k_close to close: four warps
// of work each up to 32 of them (N = 1,000: 7.5 us a call with 8 blocks, 8.1 with
// 2), then eight (N = 10,000: 8.4 us with 39 blocks, 9.4 with 78), and at most
// half of those the device holds while each warp has one slot, so that the next
// call's launch can load its tables beside this one (N = 30,000: 10.1 us with 76
// blocks, 11.0 with 117).
uint32_t single_blocks(uint32_t nslots, uint32_t resident) {
    const uint32_t half = std::max(resident / 2u, 1u), blocks = std::max(nslots / 8u, std::min(nslots / 4u, 32u));
    return std::max(1u, std::min(blocks, nslots <= half * (kSoloThreads / 32u) ? half : resident));
}

// Slots that a block of k_close lists: 64 bitmap words (16 and 32 are slower at
// N = 20,000, 9.5 us a call against 8.9; 128 at most sizes), or as many as spread
// the words over the device.
uint32_t close_slots(const spg_pop *p) {
    const uint32_t words = (p->n + 31u) / 32u, most = std::max(64u, (words + p->solo.resident - 1u) / p->solo.resident);
    return std::min(256u, (most + p->sa.slot_len - 1u) / p->sa.slot_len);
}

int launch_solo(spg_pop *p, const SoloArgs &args, const void *fn, uint32_t blocks, uint32_t threads, uint32_t smem,
                bool waits) {
    SoloArgs a = args;
    void *params[] = {&a};
    cudaLaunchAttribute attr{};
    if (waits) {  // blocks meet at a barrier, so all must be resident
        attr.id = cudaLaunchAttributeCooperative;
        attr.val.cooperative = 1;
    } else {      // its tables may load while its predecessor finishes (N = 300, one generation a call: 8.3 -> 6.5 us)
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = p->stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, params);
    return e == cudaSuccess ? SPG_OK : cuda_fail(e, "generation launch");
}

// n_gen generations: one cooperative launch per launch_gens of them.  A call
// of one generation is two launches without a barrier instead, which may start
// while their predecessors finish, as a cooperative one cannot: back to back,
// with the barrier / without, us a call: N = 3,000 10.3 / 7.8, 30,000 14.4 / 9.6,
// 10^5 16.5 / 13.8, 10^6 43.1 / 41.1.  (Two generations are no faster in pairs:
// N = 3,000 14.4 / 15.6, 30,000 16.5 / 19.2.)
int enqueue_solo(spg_pop *p, uint32_t n_gen) {
    SoloArgs a = p->sa;
    if (n_gen == 1u && p->solo_blocks > 1u) {
        a.n_gen = a.keep_last = a.single = 1u;
        a.close_slots = close_slots(p);
        const int rc = launch_solo(p, a, p->solo.fn, single_blocks(a.nslots, p->solo.resident), kSoloThreads, p->solo.smem, false);
        if (rc != SPG_OK) return rc;
        return launch_solo(p, a, close_kernel(), (a.nslots + a.close_slots - 1u) / a.close_slots, kCloseThreads, kCloseSmem,
                           false);
    }
    for (uint32_t done = 0; done < n_gen;) {
        a.n_gen = std::min(n_gen - done, p->launch_gens);
        done += a.n_gen;
        a.keep_last = done == n_gen ? 1u : 0u;
        const int rc = launch_solo(p, a, p->solo.fn, p->solo_blocks, kSoloThreads, p->solo.smem, p->solo_blocks > 1u);
        if (rc != SPG_OK) return rc;
    }
    return SPG_OK;
}

// Point the launch at the population's single segment with a launch shape
// (uploads the device copy of the segment; synchronous).
int configure_launch(spg_pop *p, const Shape &shape) {
    const PopParams &prm = *p->host_prm;
    if (!prm.continuous) {
        if (!supported_shape(p->words, shape))
            return fail(SPG_ERR_INVALID,
                        "unsupported launch shape (%u threads, %u offspring per thread, %u lanes per offspring) for %u loci",
                        shape.block, shape.items, shape.lanes, p->n_loci);
        if ((prm.linked || prm.weighted) && (shape.block != 256u || shape.items != 1u || shape.lanes != 1u))
            return fail(SPG_ERR_INVALID,
                        "a population with a linkage map or parent weights runs 256 threads, one offspring each");
        return configure_solo(p, shape);
    }
    if (shape.block != (uint32_t)kBlock || shape.items != 1u)
        return fail(SPG_ERR_INVALID, "continuous allelic values run 256 threads, one offspring each");
    OffspringKernel k = continuous_kernel(p->n_loci);
    int rc = prepare_offspring(k);
    if (rc != SPG_OK) return fail(rc, "offspring kernel setup failed");
    p->shape = shape;
    p->ntiles = (p->n + kBlock - 1) / kBlock;
    const Segment seg = segment_at(p->arena, p->L, p->n, p->ntiles, 0, p->nbuckets, 0);
    cudaError_t e = cudaMemcpyAsync(p->arena + p->L.segment, &seg, sizeof seg, cudaMemcpyHostToDevice, p->stream);
    if (e != cudaSuccess) return cuda_fail(e, "upload segment");
    rc = view_sync(p->view());
    if (rc != SPG_OK) return rc;
    p->gl = GenLaunch{};
    p->gl.offspring = k;
    p->gl.compact = compact_kernel();
    p->gl.args.segs = reinterpret_cast<const Segment *>(p->arena + p->L.segment);
    p->gl.args.one = seg;
    p->gl.args.nsegs = 1;
    p->gl.args.total_tiles = p->ntiles;
    p->gl.args.total_buckets = p->nbuckets;
    p->gl.blocks = p->ntiles;  // not persistent
    p->gl.buckets = p->nbuckets;
    p->chain.reset();
    return SPG_OK;
}

}  // namespace

extern "C" {

int spg_create_population(const spg_pop_desc *desc, const spg_allocator *alloc, void *stream, spg_pop **out) {
    if (!out) return fail(SPG_ERR_INVALID, "out is NULL");
    *out = nullptr;
    int rc = validate_desc(desc);
    if (rc != SPG_OK) return rc;
    spg_pop *p = new (std::nothrow) spg_pop();
    if (!p) return fail(SPG_ERR_OOM, "host allocation failed");
    p->n = desc->n;
    p->n_loci = desc->n_loci;
    // record = 2 * words uint32: bit-packed haplotypes, or 2L int16 values
    p->words = desc->allele_model == 1u ? desc->n_loci / 2 : desc->n_loci / 32;
    p->seed = desc->seed;
    p->rep = desc->replicate;
    p->host_prm = new (std::nothrow) PopParams();
    if (!p->host_prm) {
        delete p;
        return fail(SPG_ERR_OOM, "host allocation failed");
    }
    const bool variant = desc->map_morgans || desc->mother_weights || desc->father_weights;
    const Shape shape =
        (desc->allele_model == 1u || variant) ? Shape{(uint32_t)kBlock, 1u, 1u} : default_shape(p->words);
    rc = build_params(desc, *p->host_prm);
    if (rc != SPG_OK) {
        delete p->host_prm;
        delete p;
        return rc;
    }
    if (desc->map_morgans) rc = build_link(desc->map_morgans, p->n_loci, p->link);
    if (rc == SPG_OK && p->host_prm->weighted) {
        p->weights = new (std::nothrow) WeightParams();
        rc = p->weights ? build_weights(desc->mother_weights, desc->father_weights, *p->weights)
                        : fail(SPG_ERR_OOM, "host allocation failed");
    }
    if (rc != SPG_OK) {
        delete p->weights;
        delete p->host_prm;
        delete p;
        return rc;
    }
    p->cap = p->host_prm->stats_cap;
    p->nbuckets = bucket_count(p->n);
    if (alloc) p->alloc.hooks = *alloc;
    if (stream) {
        p->stream = (cudaStream_t)stream;
    } else {
        const cudaError_t e = cudaStreamCreateWithFlags(&p->stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) {
            delete p->host_prm;
            delete p;
            return cuda_fail(e, "cudaStreamCreate");
        }
        p->own_stream = true;
    }
    p->L = p->host_prm->continuous ? layout_for(p->n, p->words, p->nbuckets, p->cap)
                                   : solo_layout_for(p->n, p->words, p->cap, p->host_prm->weighted != 0u);
    p->arena = static_cast<char *>(p->alloc.alloc(p->L.total, p->stream));
    if (!p->arena) {
        spg_destroy(p);
        return fail(SPG_ERR_OOM, "device allocation of %zu bytes failed", p->L.total);
    }
    if (p->L.solo) {
        p->sa.dom = p->host_prm->has_dom;
        value_fragments(desc->effects, p->sa.dom ? desc->dominance : nullptr, p->n_loci, p->frag, p->sa.two_digits);
        const cudaError_t e =
            cudaMemcpyAsync(p->arena + p->L.frag, &p->frag, sizeof(ValueFragments), cudaMemcpyHostToDevice, p->stream);
        if (e != cudaSuccess) {
            spg_destroy(p);
            return cuda_fail(e, "upload value fragments");
        }
    }
    if (p->host_prm->linked) {
        p->host_prm->link = reinterpret_cast<const LinkParams *>(p->arena + p->L.link);
        const cudaError_t e =
            cudaMemcpyAsync(p->arena + p->L.link, &p->link, sizeof(LinkParams), cudaMemcpyHostToDevice, p->stream);
        if (e != cudaSuccess) {
            spg_destroy(p);
            return cuda_fail(e, "upload linkage map");
        }
    }
    if (p->host_prm->weighted) {
        p->host_prm->weights = reinterpret_cast<const WeightParams *>(p->arena + p->L.weights);
        const cudaError_t e = cudaMemcpyAsync(p->arena + p->L.weights, p->weights, sizeof(WeightParams),
                                              cudaMemcpyHostToDevice, p->stream);
        if (e != cudaSuccess) {
            spg_destroy(p);
            return cuda_fail(e, "upload parent weights");
        }
    }
    rc = view_init(p->view(), *p->host_prm,
                   desc->allele_model == 1u ? reinterpret_cast<const uint32_t *>(desc->init_values)
                                            : desc->init_genotypes,
                   desc->p0_q32);
    if (rc == SPG_OK) rc = view_sync(p->view());  // the caller's arrays are read before returning
    if (rc == SPG_OK) rc = configure_launch(p, shape);
    if (rc != SPG_OK) {
        spg_destroy(p);
        return rc;
    }
    *out = p;
    return SPG_OK;
}

int spg_set_ecology(spg_pop *p, const spg_ecology *eco) {
    if (!p) return fail(SPG_ERR_INVALID, "population is NULL");
    const int rc = view_set_ecology(p->view(), *p->host_prm, eco);
    if (rc == SPG_OK && p->L.solo) solo_args(p->view(), *p->host_prm, p->sa);
    return rc;
}

int spg_step_generations(spg_pop *p, uint32_t n_gen) {
    if (!p) return fail(SPG_ERR_INVALID, "population is NULL");
    return p->host_prm->continuous ? enqueue_generations(p->gl, n_gen, p->chain, p->stream) : enqueue_solo(p, n_gen);
}

int spg_read_stats(spg_pop *p, uint32_t first_gen, uint32_t count, spg_stats *out) {
    if (!p) return fail(SPG_ERR_INVALID, "population is NULL");
    return view_read_stats(p->view(), first_gen, count, out);
}

int spg_set_locus_counts(spg_pop *p, int enable) {
    if (!p) return fail(SPG_ERR_INVALID, "population is NULL");
    if (p->host_prm->continuous) return fail(SPG_ERR_INVALID, "per-locus allele counts are for biallelic populations");
    DevState st;
    int rc = view_state(p->view(), st);  // synchronises: no generation in flight
    if (rc != SPG_OK) return rc;
    if (enable && !p->locus_mem) {
        const uint32_t L = p->n_loci;
        const size_t ring = align_up((size_t)p->cap * L * 4u, 256), rows = (size_t)2 * L * 4u;
        p->locus_mem = static_cast<char *>(p->alloc.alloc(ring + rows, p->stream));
        if (!p->locus_mem) return fail(SPG_ERR_OOM, "device allocation of %zu bytes failed", ring + rows);
        p->locus.ring = reinterpret_cast<uint32_t *>(p->locus_mem);
        p->locus.acc = reinterpret_cast<uint32_t *>(p->locus_mem + ring);  // two rows, zero between launches
        p->locus.cap = p->cap;
        const cudaError_t e = cudaMemsetAsync(p->locus.acc, 0, rows, p->stream);
        if (e != cudaSuccess) return cuda_fail(e, "clear per-locus counts");
    }
    if (enable) {
        if (!p->locus_on) p->locus_from = st.gen + 1u;  // the first generation formed from now on
    } else if (p->locus_on) {
        p->locus_until = st.gen;  // the last generation counted
    }
    p->locus_on = enable != 0;
    attach_locus(p);
    return view_sync(p->view());
}

int spg_read_locus_counts(spg_pop *p, uint32_t first_gen, uint32_t count, uint32_t *out) {
    if (!p) return fail(SPG_ERR_INVALID, "population is NULL");
    if (!out && count) return fail(SPG_ERR_INVALID, "NULL argument");
    if (!p->locus_mem) return fail(SPG_ERR_INVALID, "per-locus allele counts are off");
    DevState st;
    const int rc = view_state(p->view(), st);
    if (rc != SPG_OK) return rc;
    if (count == 0) return SPG_OK;
    return read_locus_rows(p->locus, p->n_loci, p->locus_from, p->locus_on ? st.gen : p->locus_until, st, first_gen,
                           count, out);
}

int spg_read_genotypes(spg_pop *p, uint32_t *host, size_t n_words) {
    if (!p) return fail(SPG_ERR_INVALID, "population is NULL");
    return view_read_genotypes(p->view(), host, n_words);
}

int spg_read_survivors(spg_pop *p, uint32_t *host, size_t capacity, uint32_t *S) {
    if (!p) return fail(SPG_ERR_INVALID, "population is NULL");
    return view_read_survivors(p->view(), host, capacity, S);
}

int spg_get_state(spg_pop *p, spg_state *out) {
    if (!p) return fail(SPG_ERR_INVALID, "population is NULL");
    return view_get_state(p->view(), out);
}

int spg_checkpoint_size(spg_pop *p, size_t *bytes) {
    if (!p || !bytes) return fail(SPG_ERR_INVALID, "NULL argument");
    *bytes = sizeof(CheckpointHeader) + (size_t)p->n * 2 * p->words * 4 + (size_t)p->n * 4;
    return SPG_OK;
}

int spg_checkpoint(spg_pop *p, void *host, size_t capacity) {
    size_t need = 0;
    int rc = spg_checkpoint_size(p, &need);
    if (rc != SPG_OK) return rc;
    if (!host || capacity < need) return fail(SPG_ERR_INVALID, "checkpoint buffer too small (need %zu)", need);
    DevState st;
    rc = view_state(p->view(), st);
    if (rc != SPG_OK) return rc;
    CheckpointHeader h{};
    h.magic = kCheckpointMagic;
    h.version = SPG_ABI_VERSION;
    h.n = p->n;
    h.n_loci = p->n_loci;
    h.gen = st.gen;
    h.S = st.S;
    h.status = st.status;
    h.f = st.f;
    h.R = st.R;
    h.seed = p->seed;
    h.replicate = p->rep;
    char *dst = static_cast<char *>(host);
    std::memcpy(dst, &h, sizeof h);
    const size_t gbytes = (size_t)p->n * 2 * p->words * 4;
    cudaError_t e = cudaMemcpy(dst + sizeof h, p->arena + ((st.gen & 1u) ? p->L.geno1 : p->L.geno0), gbytes,
                               cudaMemcpyDeviceToHost);
    if (e == cudaSuccess)
        e = cudaMemcpy(dst + sizeof h + gbytes, p->arena + ((st.gen & 1u) ? p->L.surv1 : p->L.surv0),
                       (size_t)st.S * 4, cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? SPG_OK : cuda_fail(e, "checkpoint copy");
}

int spg_restore(spg_pop *p, const void *host, size_t bytes) {
    size_t need = 0;
    int rc = spg_checkpoint_size(p, &need);
    if (rc != SPG_OK) return rc;
    if (!host || bytes < sizeof(CheckpointHeader)) return fail(SPG_ERR_INVALID, "checkpoint too small");
    CheckpointHeader h;
    std::memcpy(&h, host, sizeof h);
    if (h.magic != kCheckpointMagic || h.n != p->n || h.n_loci != p->n_loci || h.S > p->n || bytes < need)
        return fail(SPG_ERR_INVALID, "checkpoint does not match this population");
    if ((h.S == 0) != (h.status == SPG_EXTINCT) || h.status < 0)
        return fail(SPG_ERR_INVALID, "checkpoint state is inconsistent");
    const char *src = static_cast<const char *>(host);
    const size_t gbytes = (size_t)p->n * 2 * p->words * 4;
    {
        // survivors index parent records: strictly increasing and < n
        const uint32_t *sv = reinterpret_cast<const uint32_t *>(src + sizeof h + gbytes);
        uint32_t prev = 0;
        for (uint32_t i = 0; i < h.S; ++i) {
            uint32_t v;
            std::memcpy(&v, sv + i, 4);
            if (v >= p->n || (i > 0 && v <= prev)) return fail(SPG_ERR_INVALID, "checkpoint survivor list is invalid");
            prev = v;
        }
    }
    rc = view_sync(p->view());
    if (rc != SPG_OK) return rc;
    // in the order of the population's stream, on which the kernels below read them
    cudaError_t e = cudaMemcpyAsync(p->arena + ((h.gen & 1u) ? p->L.geno1 : p->L.geno0), src + sizeof h, gbytes,
                                    cudaMemcpyHostToDevice, p->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p->arena + ((h.gen & 1u) ? p->L.surv1 : p->L.surv0), src + sizeof h + gbytes,
                            (size_t)h.S * 4, cudaMemcpyHostToDevice, p->stream);
    // per-bucket survivor counts of the replaced run must not leak into the
    // generations about to be replayed
    if (e == cudaSuccess && !p->L.solo)
        e = cudaMemsetAsync(p->arena + p->L.buckets, 0, (size_t)2 * p->nbuckets * 4, p->stream);
    if (e != cudaSuccess) return cuda_fail(e, "restore copy");
    if (p->L.solo) {  // the restored survivors in the slot layout: the next generation's parents
        rc = view_pack(p->view(), h.gen, reinterpret_cast<const uint32_t *>(p->arena + p->L.surv0), h.S);
        if (rc != SPG_OK) return fail(rc, "survivor packing failed");
    }
    rc = view_set_state(p->view(), h.gen, h.S, h.f, h.R, h.status, 0xFFFFFFFFu);
    if (rc != SPG_OK) return rc;
    if (p->locus_mem) {  // the rows of a generation that failed hold part of its counts
        e = cudaMemsetAsync(p->locus.acc, 0, (size_t)2 * p->n_loci * 4, p->stream);
        if (e != cudaSuccess) return cuda_fail(e, "clear per-locus counts");
    }
    p->locus_from = h.gen + 1u;  // counts of the restored run start with its next generation
    p->locus_until = h.gen;
    return view_sync(p->view());
}

int spg_set_tiling(spg_pop *p, uint32_t items) {
    spg_launch_shape sh{256u, items, 1u};
    return spg_set_launch_shape(p, &sh);
}

int spg_get_tiling(spg_pop *p, uint32_t *items) {
    if (!p || !items) return fail(SPG_ERR_INVALID, "NULL argument");
    *items = p->shape.items;
    return SPG_OK;
}

int spg_set_launch_shape(spg_pop *p, const spg_launch_shape *shape) {
    if (!p || !shape) return fail(SPG_ERR_INVALID, "NULL argument");
    Shape sh;
    int rc = shape_from_abi(p->host_prm->continuous ? 0u : p->words, shape, sh);
    if (rc != SPG_OK) return rc;
    rc = view_sync(p->view());
    if (rc != SPG_OK) return rc;
    return configure_launch(p, sh);
}

int spg_get_launch_shape(spg_pop *p, spg_launch_shape *out) {
    if (!p || !out) return fail(SPG_ERR_INVALID, "NULL argument");
    out->threads_per_block = p->shape.block;
    out->items_per_thread = p->shape.items;
    out->lanes_per_offspring = p->shape.lanes;
    return SPG_OK;
}

int spg_synchronize(spg_pop *p) {
    if (!p) return fail(SPG_ERR_INVALID, "population is NULL");
    return view_sync(p->view());
}

void spg_destroy(spg_pop *p) {
    if (!p) return;
    if (p->stream) cudaStreamSynchronize(p->stream);
    p->chain.reset();
    if (p->locus_mem) p->alloc.release(p->locus_mem, p->stream);
    if (p->arena) p->alloc.release(p->arena, p->stream);
    if (p->stream) cudaStreamSynchronize(p->stream);
    if (p->own_stream && p->stream) cudaStreamDestroy(p->stream);
    delete p->weights;
    delete p->host_prm;
    delete p;
}

}  // extern "C"
