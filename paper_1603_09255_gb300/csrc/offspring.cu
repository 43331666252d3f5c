// The offspring kernel of the allocation-free generation call (sm_103a):
// Fig. 1 A-D of the paper for every offspring of one population whose buffers
// the caller owns, the previous survivors given as a list of indices.  (The
// library's own populations keep their survivors' records packed and are
// formed by generations.cuh.)
//
// Persistent: each block forms one contiguous share of the population's
// tiles.  Per offspring it draws both parents from the previous survivors
// (A), forms the gametes by crossover masks and mutation XOR (B), sums the
// genetic value (C) and decides survival (D); it writes the child record, the
// alive bitmap, per-bucket survivor counts and exact integer statistics.
//
// A parent is a survivor index read by rank and then its record, a single
// vector load (256 bits for L = 128, two for L = 256): random reads are
// bounded by the number of L2 requests, and one request per 32-byte sector is
// the minimum.  The records of tile t+1 are loaded into registers while tile
// t is formed, the draws and indices of tile t+2 made before that.
//
// The block copies the survival thresholds by phenotype bin and the byte
// tables of the genetic value into its dynamic shared memory with cp.async:
// entry (k, v) of the latter is the sum of the effects of loci 8k .. 8k+7
// whose allele bit is set in v, so a haplotype's additive value is L/8
// shared-memory lookups instead of a popcount per effect bit plane and word
// (a popcount issues at a quarter of the integer rate).
//
// L <= 128: one thread per offspring, tiles of 256.  L = 256: two lanes per
// offspring (see lane pairs), tiles of 128.
#include "device_common.cuh"

namespace spg {
namespace {

constexpr int kThreads = 256;
constexpr int kBlocksPerSM = 2;  // the register cap: 16 warps per SM
constexpr int NW = kThreads / 32;
template <int W>
constexpr uint32_t kTile = W == 8 ? kThreads / 2 : kThreads;  // offspring per tile

// The population as the tile loop sees it.
struct SegCtx {
    const uint32_t *par;  // parent records by index
    const uint32_t *sin;  // survivor indices
    uint32_t *chi;
    uint32_t *alive;
    uint32_t *bucket_now;
    uint32_t n, S, f, g, rep, k0, k1, kmax, shift;
    int32_t bias;
};

// The dynamic shared memory: the byte tables of the additive value at 0 (so a
// lookup's address is its byte value times 4 plus a constant), the survival
// thresholds after them.
extern __shared__ __align__(16) unsigned char s_dyn[];
template <int W>
struct SmemLayout {
    static constexpr uint32_t kThr = 4096u * W;  // 4W byte tables of 256 int32
    static constexpr uint32_t kBytes = kThr + kBins * 4u;
};

__device__ __forceinline__ uint32_t smem_u32(uint32_t byte_off) {
    return *reinterpret_cast<const uint32_t *>(s_dyn + byte_off);
}
__device__ __forceinline__ int32_t smem_i32(uint32_t byte_off) {
    return *reinterpret_cast<const int32_t *>(s_dyn + byte_off);
}

// One parent record (2W words) in a single request per 32-byte sector,
// through L2 only (the parents are read-only for the whole launch).
template <int W>
__device__ __forceinline__ void load_parent(const uint32_t *__restrict__ p, uint32_t (&r)[2 * W]) {
    if constexpr (W == 1) {
        asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "l"(p));
    } else if constexpr (W == 2) {
        asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "l"(p));
    } else {
#pragma unroll
        for (int q = 0; q < W / 4; ++q)
            asm volatile("ld.global.nc.L1::no_allocate.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(r[8 * q]), "=r"(r[8 * q + 1]), "=r"(r[8 * q + 2]), "=r"(r[8 * q + 3]),
                           "=r"(r[8 * q + 4]), "=r"(r[8 * q + 5]), "=r"(r[8 * q + 6]), "=r"(r[8 * q + 7])
                         : "l"(p + 8 * q));
    }
}

// Sum of the byte-table entries of one word x holding loci 32w .. 32w+31 (its
// four bytes): part of a haplotype's genetic value (eq. S2-phenval, per locus
// e_l * allele), exact in int32.
__device__ __forceinline__ int32_t byte_table_word(uint32_t w, uint32_t x) {
    constexpr uint32_t T = (uint32_t)kLutWords * 4u;  // bytes per table
    const uint32_t t = 4u * w * T;
    return smem_i32(t + ((x << 2) & 0x3FCu)) + smem_i32(t + T + ((x >> 6) & 0x3FCu)) +
           smem_i32(t + 2u * T + ((x >> 14) & 0x3FCu)) + smem_i32(t + 3u * T + ((x >> 22) & 0x3FCu));
}

struct ThreadStats {
    long long sum_raw = 0, sum_raw_s = 0;
    unsigned long long sum_raw2 = 0;
    uint32_t het = 0, allele = 0;
    int mn = INT_MAX, mx = INT_MIN;
};

// (D) survival: the bin's threshold scaled by the resource factor; the
// offspring's statistics.
template <int W>
__device__ __forceinline__ bool survives(const SegCtx &c, int32_t raw, uint32_t u_surv) {
    const long long v = (long long)raw + (long long)c.bias;
    const uint32_t bin = v < 0 ? 0u : (uint32_t)min(v >> c.shift, (long long)(kBins - 1));
    uint32_t thr = smem_u32(SmemLayout<W>::kThr + bin * 4u);
    if (c.f != kCertain) thr = __umulhi(thr, c.f);
    return (thr == kCertain) || (u_surv < thr);
}
__device__ __forceinline__ void add_value(ThreadStats &ts, int32_t raw, bool alive) {
    ts.sum_raw += raw;
    ts.sum_raw2 += (unsigned long long)((long long)raw * (long long)raw);
    ts.mn = min(ts.mn, raw);
    ts.mx = max(ts.mx, raw);
    if (alive) ts.sum_raw_s += raw;
}

// Mutations of an offspring from its draw (none below the CDF's first entry,
// the common case).
__device__ __forceinline__ uint32_t mutations(const SegCtx &c, const uint32_t *s_cdf, uint32_t u_mut) {
    uint32_t k = 0;
    if (c.kmax != 0u && u_mut >= s_cdf[0])
        for (uint32_t i = 0; i < c.kmax; ++i) k += (u_mut >= s_cdf[i]) ? 1u : 0u;
    return k;
}

// ------------------------------------------------ one thread per offspring
template <int W>
struct Single {
    struct Draws {
        uint32_t mom, dad, u_surv, u_mut;  // record indices; the survival and mutation-count draws
    };
    struct Recs {
        uint32_t m[2 * W], f[2 * W];
    };

    static __device__ __forceinline__ void draw(const SegCtx &c, uint32_t base, int tid, Draws &d) {
        const uint32_t j = base + (uint32_t)tid;
        d.mom = d.dad = d.u_surv = d.u_mut = 0u;
        if (j < c.n) {
            const uint4 r = philox(make_uint4(j, c.g, c.rep, kMate << 24), c.k0, c.k1);
            // survivor indices through L2 only (random 4-byte reads)
            d.mom = __ldcg(c.sin + __umulhi(r.x, c.S));
            d.dad = __ldcg(c.sin + __umulhi(r.y, c.S));
            d.u_surv = r.z;
            d.u_mut = r.w;
        }
    }

    static __device__ __forceinline__ void load(const SegCtx &c, uint32_t base, int tid, const Draws &d, Recs &rec) {
        if (base + (uint32_t)tid < c.n) {
            load_parent<W>(c.par + (size_t)d.mom * (2 * W), rec.m);
            load_parent<W>(c.par + (size_t)d.dad * (2 * W), rec.f);
        }
    }

    // One tile: gametes (B), genetic value (C), survival (D), bitmap (E, first
    // half); returns the warp's survivors.
    static __device__ __forceinline__ uint32_t tile(const SegCtx &c, uint32_t base, int tid, int lane, int warp,
                                                    const Recs &rec, const Draws &dr, const uint32_t *s_cdf,
                                                    ThreadStats &ts) {
        const uint32_t j = base + (uint32_t)tid;
        bool alive = false;
        if (j < c.n) {
            uint32_t ch[2 * W];
            // (B) gametes: stream q = 2w + parent is lane q%4 of sub q/4
#pragma unroll
            for (int q4 = 0; q4 < (2 * W + 3) / 4; ++q4) {
                const uint4 d = philox(make_uint4(j, c.g, c.rep, (kRecomb << 24) | (uint32_t)q4), c.k0, c.k1);
#pragma unroll
                for (int l = 0; l < 4; ++l) {
                    const int q = 4 * q4 + l;
                    if (q < 2 * W) {
                        const int w = q >> 1;
                        const uint32_t m = lane_of(d, l);
                        if ((q & 1) == 0) ch[w] = (rec.m[w] & ~m) | (rec.m[W + w] & m);
                        else ch[W + w] = (rec.f[w] & ~m) | (rec.f[W + w] & m);
                    }
                }
            }
            const uint32_t k = mutations(c, s_cdf, dr.u_mut);
            if (k) mutate<W>(ch, k, j, c.g, c.rep, c.k0, c.k1);
            store_record<W>(c.chi + (size_t)j * (2 * W), ch);
            // (C) genetic value from the byte tables
            int32_t raw = 0;
            uint32_t allele = 0, hz = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                raw += byte_table_word((uint32_t)w, ch[w]) + byte_table_word((uint32_t)w, ch[W + w]);
                allele += __popc(ch[w]) + __popc(ch[W + w]);
                hz += __popc(ch[w] ^ ch[W + w]);
            }
            alive = survives<W>(c, raw, dr.u_surv);
            add_value(ts, raw, alive);
            ts.het += hz;
            ts.allele += allele;
        }
        // (E, first half) alive bitmap word (base + 32*warp)/32
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, alive);
        if (lane == 0) c.alive[(base >> 5) + (uint32_t)warp] = bal;
        return __popc(bal);
    }
};

// ----------------------------------------------------------- lane pairs
// L = 256: two lanes per offspring.  Lane h of a pair (h = 0 mother, 1
// father) draws that parent, loads its record (one request per sector) and
// forms the gamete that becomes the child's haplotype h; the pair shares the
// gamete-mask draws (each lane computes half the Philox blocks and hands the
// other lane its lanes of them), the genetic value (each lane sums its
// gamete's byte tables) and the survival decision.  A lane holds one parent
// record instead of two (two do not fit a thread's registers twice over); the
// two gametes of a child are written by adjacent lanes as one coalesced
// record.
// The gamete-mask words of lane h's parent: the gamete stream q = 2w + h is
// lane q % 4 of Philox sub q / 4 (sub s covers words 2s and 2s+1: lanes x, y
// mother and father of word 2s, z, w of word 2s+1).  Of each pair of subs
// (2t, 2t+1) lane h computes sub 2t + h and receives its lanes of the other
// from the partner lane.  All lanes of the warp take part (shuffles).
template <int W>
__device__ __forceinline__ void pair_masks(const SegCtx &c, uint32_t j, uint32_t h, uint32_t (&m)[W]) {
    static_assert(W % 4 == 0, "lane pairs serve records of 4 or 8 words per haplotype");
#pragma unroll
    for (int t = 0; t < W / 4; ++t) {
        const uint4 d = philox(make_uint4(j, c.g, c.rep, (kRecomb << 24) | (uint32_t)(2 * t) + h), c.k0, c.k1);
        const uint32_t a = __shfl_xor_sync(0xFFFFFFFFu, h ? d.x : d.y, 1);
        const uint32_t b = __shfl_xor_sync(0xFFFFFFFFu, h ? d.z : d.w, 1);
        m[4 * t + 0] = h ? a : d.x;  // word 4t:   sub 2t, lane x (mother) / y (father)
        m[4 * t + 1] = h ? b : d.z;  // word 4t+1: sub 2t, lane z / w
        m[4 * t + 2] = h ? d.y : a;  // word 4t+2: sub 2t+1, lane x / y
        m[4 * t + 3] = h ? d.w : b;  // word 4t+3: sub 2t+1, lane z / w
    }
}

// Per-locus mutation of a pair's child (the draws of mutate(), made by both
// lanes alike): each position belongs to one haplotype, whose lane checks it
// against the positions already chosen there and flips it; the pair agrees
// on every duplicate through a shuffle, so both count the same K distinct
// positions.
template <int W>
__device__ __forceinline__ void pair_mutate(uint32_t (&g)[W], uint32_t k, uint32_t j, uint32_t gen, uint32_t rep,
                                            uint32_t k0, uint32_t k1, uint32_t h, uint32_t pair_mask) {
    constexpr uint32_t L = 32u * W;
    uint32_t seen[W];
#pragma unroll
    for (int w = 0; w < W; ++w) seen[w] = 0u;
    uint32_t chosen = 0;
    for (uint32_t a4 = 0; a4 < kMutDraws / 4 && chosen < k; ++a4) {
        const uint4 d = philox(make_uint4(j, gen, rep, (kMutPos << 24) | a4), k0, k1);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            if (chosen < k) {
                const uint32_t pos = __umulhi(lane_of(d, l), 2u * L);  // [0, 2L)
                const uint32_t owner = pos >= L ? 1u : 0u, loc = pos - owner * L;
                const uint32_t wi = loc >> 5, bit = 1u << (loc & 31u);
                bool mine_dup = false;
#pragma unroll
                for (int w = 0; w < W; ++w)
                    if ((uint32_t)w == wi) mine_dup = (seen[w] & bit) != 0u;
                const bool other_dup = __shfl_xor_sync(pair_mask, mine_dup, 1);
                const bool dup = owner == h ? mine_dup : other_dup;
                if (!dup) {
                    if (owner == h) {
#pragma unroll
                        for (int w = 0; w < W; ++w)
                            if ((uint32_t)w == wi) {
                                seen[w] |= bit;
                                g[w] ^= bit;
                            }
                    }
                    ++chosen;
                }
            }
        }
    }
}

// The W words of a gamete at p (32-byte aligned).
__device__ __forceinline__ void store_gamete(uint32_t *__restrict__ p, const uint32_t (&g)[8]) {
    asm volatile("st.global.v8.u32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(g[0]), "r"(g[1]), "r"(g[2]),
                 "r"(g[3]), "r"(g[4]), "r"(g[5]), "r"(g[6]), "r"(g[7]));
}

template <int W>
struct Pair {
    struct Draws {
        uint32_t par, u_surv, u_mut;  // this lane's parent, the offspring's uniforms
    };
    struct Recs {
        uint32_t r[2 * W];  // this lane's parent record
    };

    static __device__ __forceinline__ void draw(const SegCtx &c, uint32_t base, int tid, Draws &d) {
        const uint32_t j = base + (uint32_t)(tid >> 1);
        d.par = d.u_surv = d.u_mut = 0u;
        if (j < c.n) {
            const uint4 r = philox(make_uint4(j, c.g, c.rep, kMate << 24), c.k0, c.k1);
            d.par = __ldcg(c.sin + __umulhi((tid & 1) ? r.y : r.x, c.S));
            d.u_surv = r.z;
            d.u_mut = r.w;
        }
    }

    static __device__ __forceinline__ void load(const SegCtx &c, uint32_t base, int tid, const Draws &d, Recs &rec) {
        if (base + (uint32_t)(tid >> 1) < c.n) load_parent<W>(c.par + (size_t)d.par * (2 * W), rec.r);
    }

    static __device__ __forceinline__ uint32_t tile(const SegCtx &c, uint32_t base, int tid, int lane, int warp,
                                                    const Recs &rec, const Draws &dr, const uint32_t *s_cdf,
                                                    ThreadStats &ts) {
        const uint32_t h = (uint32_t)lane & 1u, pair_mask = 3u << (lane & ~1);
        const uint32_t j = base + (uint32_t)(tid >> 1);
        const bool live = j < c.n;
        // (B) this lane's gamete from its parent: crossover masks, mutation
        uint32_t m[W], g[W];
        pair_masks<W>(c, j, h, m);
#pragma unroll
        for (int w = 0; w < W; ++w) g[w] = (rec.r[w] & ~m[w]) | (rec.r[W + w] & m[w]);
        const uint32_t k = live ? mutations(c, s_cdf, dr.u_mut) : 0u;  // the same in both lanes of the pair
        if (k) pair_mutate<W>(g, k, j, c.g, c.rep, c.k0, c.k1, h, pair_mask);
        if (live) store_gamete(c.chi + (size_t)j * (2 * W) + h * W, g);
        // (C) genetic value: this gamete's additive value; the heterozygosity
        // of half of the words
        int32_t part = 0;
        uint32_t allele = 0, hz = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            part += byte_table_word((uint32_t)w, g[w]);
            allele += __popc(g[w]);
        }
#pragma unroll
        for (int i = 0; i < W / 2; ++i) {
            const uint32_t mine = h ? g[W / 2 + i] : g[i];  // words h * W/2 + i
            const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, h ? g[i] : g[W / 2 + i], 1);
            hz += __popc(mine ^ other);
        }
        const int32_t raw = part + __shfl_xor_sync(0xFFFFFFFFu, part, 1);
        bool alive = false;
        if (live) {
            alive = survives<W>(c, raw, dr.u_surv);
            ts.het += hz;
            ts.allele += allele;
            if (h == 0u) add_value(ts, raw, alive);  // the offspring's sums once per pair
        }
        // (E, first half) the warp's 16 offspring: bit p of the half word is
        // pair p's decision (the even lanes of the ballot)
        uint32_t bal = __ballot_sync(0xFFFFFFFFu, alive) & 0x55555555u;
        bal = (bal | (bal >> 1)) & 0x33333333u;
        bal = (bal | (bal >> 2)) & 0x0F0F0F0Fu;
        bal = (bal | (bal >> 4)) & 0x00FF00FFu;
        bal = (bal | (bal >> 8)) & 0x0000FFFFu;
        const uint32_t j0 = base + (uint32_t)(warp * 16);
        if (lane == 0) reinterpret_cast<uint16_t *>(c.alive)[j0 >> 4] = (uint16_t)bal;
        return __popc(bal);
    }
};

// Tiles [lt0, lt1) of the population (see the file comment for the pipeline).
template <int W, typename Form>
__device__ __forceinline__ void form_tiles(const SegCtx &c, uint32_t lt0, uint32_t lt1, uint32_t *bucket_next, int tid,
                                           int lane, int warp, const uint32_t *s_cdf, ThreadStats &ts,
                                           uint32_t &warp_alive) {
    constexpr uint32_t TILE = kTile<W>;
    typename Form::Draws d0, d1;
    typename Form::Recs ra, rb;
    Form::draw(c, lt0 * TILE, tid, d0);
    if (lt0 + 1 < lt1) Form::draw(c, (lt0 + 1) * TILE, tid, d1);
    Form::load(c, lt0 * TILE, tid, d0, ra);
    cp_async_wait<0>();
    __syncthreads();  // the tables (and cdf) are visible to every thread

    uint32_t bucket_alive = 0, bucket_cur = (lt0 * TILE) / kBucket;
    // one tile: prefetch the next tile's records, draw the one after next
    // (before forming this one, so the compiler can interleave its Philox
    // rounds with the tile's), form this one
    auto step = [&](uint32_t lt, const typename Form::Recs &cur, typename Form::Recs &nxt) {
        const uint32_t base = lt * TILE;
        if (lt + 1 < lt1) Form::load(c, base + TILE, tid, d1, nxt);
        if (tid == 0 && base % kBucket == 0u) bucket_next[base / kBucket] = 0u;
        const uint32_t bkt = base / kBucket;
        if (bkt != bucket_cur) {
            if (lane == 0 && bucket_alive) atomicAdd(&c.bucket_now[bucket_cur], bucket_alive);
            bucket_alive = 0;
            bucket_cur = bkt;
        }
        typename Form::Draws d2;
        Form::draw(c, base + 2 * TILE, tid, d2);  // past the share: unused
        const uint32_t cnt = Form::tile(c, base, tid, lane, warp, cur, d0, s_cdf, ts);
        bucket_alive += cnt;
        warp_alive += cnt;
        d0 = d1;
        d1 = d2;
    };
    for (uint32_t lt = lt0; lt < lt1; lt += 2) {  // record sets alternate, so no register copies
        step(lt, ra, rb);
        if (lt + 1 < lt1) step(lt + 1, rb, ra);
    }
    if (lane == 0 && bucket_alive) atomicAdd(&c.bucket_now[bucket_cur], bucket_alive);
}

template <int W, typename Form>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM) k_offspring(const __grid_constant__ GenArgs a) {
    static_assert(kBucket % kTile<W> == 0, "tiles must not straddle compaction buckets");
    __shared__ uint32_t s_cdf[kMaxKmax];
    __shared__ long long s_ll[2][NW];
    __shared__ unsigned long long s_ull[NW];
    __shared__ uint32_t s_u32[3][NW];
    __shared__ int s_mm[2][NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t dyn = (uint32_t)__cvta_generic_to_shared(s_dyn);
    const Segment &sg = a.one;
    const uint32_t T = a.total_tiles, G = gridDim.x;
    const uint32_t lt0 = (uint32_t)(((unsigned long long)T * blockIdx.x) / G);
    const uint32_t lt1 = (uint32_t)(((unsigned long long)T * (blockIdx.x + 1)) / G);
    // the tables (parameters only: nothing the previous kernel writes)
    const PopParams *P = sg.prm;
    constexpr uint32_t kTab16 = (uint32_t)kBins * 4u / 16u;         // 16-byte chunks of the bin table
    constexpr uint32_t kLut16 = (uint32_t)W * 4u * kLutWords / 4u;  // of the 4W byte tables
    for (uint32_t i = (uint32_t)tid; i < kTab16; i += kThreads)
        cp_async_16(dyn + SmemLayout<W>::kThr + 16u * i, P->table + 4u * i);
    for (uint32_t i = (uint32_t)tid; i < kLut16; i += kThreads) cp_async_16(dyn + 16u * i, P->lut + 4u * i);
    cp_async_commit();
    if (tid < kMaxKmax) s_cdf[tid] = (uint32_t)tid < P->kmax ? P->cdf[tid] : 0u;
    griddep_wait();  // from here on: the previous kernel's state, records and counters
    const PopNow now = read_state(sg.state);
    if (lt0 < lt1 && now.active) {
        SegCtx c;
        c.n = sg.n;
        c.S = min(now.S, sg.n);  // parent ranks stay inside the buffers whatever the state holds
        c.f = now.f;
        c.g = now.gen + 1u;
        c.sin = sg.surv[now.gen & 1u];
        c.par = sg.geno[now.gen & 1u];
        c.chi = sg.geno[(now.gen + 1u) & 1u];
        c.alive = sg.alive;
        c.bucket_now = sg.bucket_sum + (c.g & 1u) * sg.nbuckets;
        uint32_t *bucket_next = sg.bucket_sum + ((c.g + 1u) & 1u) * sg.nbuckets;
        c.rep = P->rep;
        c.k0 = P->key0;
        c.k1 = P->key1;
        c.kmax = P->kmax;
        c.shift = P->shift;
        c.bias = P->bias;
        ThreadStats ts;
        uint32_t warp_alive = 0;
        form_tiles<W, Form>(c, lt0, lt1, bucket_next, tid, lane, warp, s_cdf, ts, warp_alive);

        // statistics of this share: exact warp sums, one atomic per field into
        // one of the population's accumulator copies
        const long long w_raw = warp_sum_i64(ts.sum_raw), w_raw_s = warp_sum_i64(ts.sum_raw_s);
        const unsigned long long w_raw2 = warp_sum_u64(ts.sum_raw2);
        const uint32_t w_het = __reduce_add_sync(0xFFFFFFFFu, ts.het);
        const uint32_t w_allele = __reduce_add_sync(0xFFFFFFFFu, ts.allele);
        const int w_mn = __reduce_min_sync(0xFFFFFFFFu, ts.mn), w_mx = __reduce_max_sync(0xFFFFFFFFu, ts.mx);
        if (lane == 0) {
            s_ll[0][warp] = w_raw;
            s_ll[1][warp] = w_raw_s;
            s_ull[warp] = w_raw2;
            s_u32[0][warp] = w_het;
            s_u32[1][warp] = w_allele;
            s_u32[2][warp] = warp_alive;
            s_mm[0][warp] = w_mn;
            s_mm[1][warp] = w_mx;
        }
        __syncthreads();
        if (tid == 0) {
            long long a0 = 0, a1 = 0;
            unsigned long long b0 = 0, hz = 0, al = 0, sv = 0;
            int m0 = INT_MAX, m1 = INT_MIN;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                a0 += s_ll[0][w];
                a1 += s_ll[1][w];
                b0 += s_ull[w];
                hz += s_u32[0][w];
                al += s_u32[1][w];
                sv += s_u32[2][w];
                m0 = min(m0, s_mm[0][w]);
                m1 = max(m1, s_mm[1][w]);
            }
            StatAcc *acc = sg.acc + blockIdx.x % kAccCopies;
            atomicAdd(&acc->s, sv);
            atomicAdd(reinterpret_cast<unsigned long long *>(&acc->sum_raw), (unsigned long long)a0);
            atomicAdd(reinterpret_cast<unsigned long long *>(&acc->sum_raw_s), (unsigned long long)a1);
            atomicAdd(&acc->sum_raw2, b0);
            atomicAdd(&acc->het, hz);
            atomicAdd(&acc->allele, al);
            atomicMin(&acc->mn, m0);
            atomicMax(&acc->mx, m1);
        }
    } else {
        cp_async_wait<0>();  // the tables' copies have landed before the block's memory goes away
    }
    // the compaction's blocks are launched once every block of this grid is
    // here (released at entry instead, they took SM resources from this
    // grid's tail: 5% slower generations)
    griddep_release();
}

template <int W, typename Form>
OffspringKernel instance() {
    OffspringKernel k;
    k.fn = &k_offspring<W, Form>;
    k.tile = kTile<W>;
    k.smem = SmemLayout<W>::kBytes;
    k.programmatic = true;
    return k;
}

}  // namespace

OffspringKernel offspring_kernel(uint32_t words) {
    switch (words) {
        case 1: return instance<1, Single<1>>();
        case 2: return instance<2, Single<2>>();
        case 4: return instance<4, Single<4>>();
        case 8: return instance<8, Pair<8>>();
        default: return OffspringKernel{};
    }
}

}  // namespace spg
