// The generation kernel of biallelic populations (sm_103a): any number of
// generations of Fig. 1 A-F in one cooperative launch, of one population
// (k_generations) or of many of a kind, each formed by a team of blocks (k_teams).
//
// us per generation, against an offspring launch with byte tables and a
// compaction launch: N = 10^4, L = 32: 8.2 -> 4.8; 99,991 x 64 with locus counts
// 21.5 -> 9.9; 3 x 10^5 x 128 with dominance 23.8 -> 13.2; 10^6 x 128 with a
// resource 39.2 -> 26.1, with a map 127 -> 74, with weights 64.8 -> 48.5; 2 x
// 10^6 x 256 164 -> 78.  At 10^6 x 128 it is bound by instructions: 479 per warp
// of 32 offspring in a launch of four generations, of which some 400 form the
// offspring (41,000 of 52,000 cycles of a generation); the ALU pipe is busy 46 %
// of the cycles and an instruction issues in 44 % of them, with four warps per
// scheduler (512 threads of 128 registers; 640 to 1,024 threads spill and are
// slower).  The rest is the barrier (3,300 to 5,000 cycles), the directory (2,000
// to 3,500) and the statistics.
//
// Blocks stay for the whole call, so the tables (thresholds, attack rates,
// effect digits, linkage map) reach shared memory once per call instead of
// once per launch and generation, and a generation costs one grid barrier.
//
// Slots.  The population's groups of 32 offspring are cut into at most
// 152 slots a warp of equal length, one per resident warp at large N.  A warp
// forms its slot's groups in order and packs the survivors' records at the
// start of the slot's own range, counting them; no other pass touches a
// record.  Between generations every block turns the slots' counts into a
// directory in its shared memory: slot s holds the survivors of ranks
// P[s] .. P[s+1]-1 (index order, as slots are contiguous), at record
// s * 32 * slot_len + (rank - P[s]).  A parent's rank finds its slot through a
// guide by the draw's top bits and about a quarter of a step forward.  This replaces
// a compaction launch that read every child and rewrote the survivors.
//
// Full records, the survivor bitmap and the ordered survivor list are only
// visible between calls, so they are written in a call's last generation
// (and in one that leaves no survivors: it is formed a second time for them).
// The per-locus counts read full records, so those are written every
// generation while counting.  A call of one generation has no barrier: k_close
// (kernels.cu) closes what this kernel has formed.
//
// Genetic value.  A child's value is a counts x effects product: the warp's 32
// records go through shared memory into mma.m16n8k16 fragments, each locus as
// an f16 element.  The two haplotypes' bits of a locus are brought side by
// side as a 2-bit count (carry-save: x = h0 ^ h1, 2 (h0 & h1)), and a count at
// bits p, p+1 of a half word IS the f16 number count * 2^(p-24) for p <= 10
// (subnormals and the first two binades are linear), so a mask makes two
// elements: no conversion.  The effects (exact f16, |e| <= 2048) are scaled to
// undo 2^p; every product is a multiple of 2^-20 and the sums stay below 2^22
// of them: exact in the fp32 accumulators.  Even columns hold the effects for
// every q, odd columns ones (the allele count), so each lane finds its own
// offspring's sums without a shuffle; larger effects are two digits of radix
// 2048 in the even and odd columns.  With dominance the elements are x (value
// e + d) and h0 & h1 (value 2e) apart.  (e4m3 elements, four to a word, are
// taken apart into f16 by this target: 2.4 times the instructions.)
#pragma once

#include "closing.cuh"

namespace spg {
namespace {

// ------------------------------------------------------- shared memory
constexpr uint32_t kGuide = 1u << kMaxGuideBits;  // most entries of the guide

template <int W, bool LINKED>
struct GenSmem {
    static constexpr uint32_t BLOCK = kSoloThreads, kSlots = kMaxSlots;
    static constexpr uint32_t NW = BLOCK / 32;
    static constexpr uint32_t kPlanes = W <= 2 ? 1u : (uint32_t)W / 2u;  // 16-byte planes of a staged record
    static constexpr uint32_t kSets = W == 8 ? 2u : 1u;                  // word sets of the value fragments
    static constexpr uint32_t kRegs = W >= 4 ? 16u : 4u * W;             // element pairs of a lane, row and set
    static constexpr uint32_t kRegRoom = kRegs < 8u ? 8u : kRegs;        // places for them (even loci, odd loci)
    static constexpr uint32_t kThr = 0u, kAtt = kThr + kBins * 4u, kDir = kAtt + kBins * 4u;
    static constexpr uint32_t kGuideOff = kDir + kSlots * 8u;
    static constexpr uint32_t kFrag = kGuideOff + kGuide * 2u;           // [table][set][kRegRoom / 4][32][4]
    static constexpr uint32_t kSetBytes = kRegRoom * 128u, kTabBytes = kSets * kSetBytes;
    static constexpr uint32_t kStage = kFrag + 2u * kTabBytes;
    static constexpr uint32_t kRecStage = kPlanes * 512u;
    static constexpr uint32_t kTog = LINKED ? 2u * 32u * (uint32_t)W * 4u : 0u;
    static constexpr uint32_t kPerWarp = kRecStage > kTog ? kRecStage : (kTog + 15u) / 16u * 16u;
    static constexpr uint32_t kLinkOff = kStage + NW * kPerWarp;
    // linkage map: cdf, cum, guide, first
    static constexpr uint32_t kLinkBytes = LINKED ? kMaxKmax * 4u + kMaxLoci * 4u + kLinkGuide * 4u + (kMaxChrom + 2u) * 2u : 0u;
    static constexpr uint32_t kThreads = BLOCK;
    static constexpr uint32_t kStats = (kLinkOff + kLinkBytes + 15u) / 16u * 16u;  // lanes' statistics, 48 bytes each
    static constexpr uint32_t kBytes = kStats + 48u * BLOCK;
};

extern __shared__ __align__(128) unsigned char g_smem[];

__device__ __forceinline__ uint32_t sm_u32(uint32_t off) { return *reinterpret_cast<const uint32_t *>(g_smem + off); }

// ------------------------------------------------------- team barrier
// All blocks of a population's team (a cooperative grid's blocks, or some of
// them) arrive and wait; false when the wait ran out.  The counter only grows,
// by kBarrierStep per barrier whatever the team's size (its first block adds
// what the others leave).  (Every block polling a word of every other took 5 us
// instead of 2 with 152 blocks.)
//
// A block whose polls run out marks the counter, in one atomic step and only
// while the barrier is incomplete: from then on nobody passes it, however late
// the missing blocks arrive, so the generation is closed by nobody and every
// block of the team reports the failure.  The mark stays until the population's
// memory is set up again (launch_pack).
constexpr unsigned long long kBarrierStep = 1u << 16;  // more than a grid's blocks
constexpr unsigned long long kBarrierFailed = 1ull << 63;

// The end of a wait whose polls ran out, or that met the mark: whether the
// barrier was complete after all.
__device__ __noinline__ int barrier_given_up(unsigned long long *ctr, unsigned long long v, unsigned long long want) {
    while (v < want && v < kBarrierFailed) {  // once per arrival meanwhile, at most
        const unsigned long long was = atomicCAS(ctr, v, v | kBarrierFailed);
        v = was == v ? kBarrierFailed : was;
    }
    return v < kBarrierFailed ? 1 : 0;
}

__device__ __forceinline__ bool team_barrier(unsigned long long *ctr, uint32_t rank, uint32_t team, uint32_t tries) {
    __syncthreads();
    if (team == 1u) return true;
    int ok = 1;
    if (threadIdx.x == 0) {
        const unsigned long long add = rank == 0u ? kBarrierStep - (team - 1u) : 1ull;
        unsigned long long old;
        asm volatile("atom.add.release.gpu.global.u64 %0, [%1], %2;" : "=l"(old) : "l"(ctr), "l"(add) : "memory");
        const unsigned long long want = (old / kBarrierStep + 1ull) * kBarrierStep;
        unsigned long long v = old < kBarrierFailed ? 0ull : ~0ull;  // (a marked barrier is not waited for)
        for (uint32_t i = 0; i < tries && v < want; ++i)
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(ctr) : "memory");
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        if (v < want || v >= kBarrierFailed) ok = barrier_given_up(ctr, v, want);
    }
    return __syncthreads_and(threadIdx.x == 0 ? ok : 1) != 0;
}

// ------------------------------------------------------- record access
// Parents are read through L2: their buffers change during the launch.
template <int W>
__device__ __forceinline__ void load_packed(const uint32_t *p, uint32_t (&r)[2 * W]) {
    if constexpr (W == 1) {
        asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "l"(p) : "memory");
    } else if constexpr (W == 2) {
        asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "l"(p) : "memory");
    } else {
#pragma unroll
        for (int q = 0; q < W / 4; ++q)
            asm volatile("ld.global.cg.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(r[8 * q]), "=r"(r[8 * q + 1]), "=r"(r[8 * q + 2]), "=r"(r[8 * q + 3]),
                           "=r"(r[8 * q + 4]), "=r"(r[8 * q + 5]), "=r"(r[8 * q + 6]), "=r"(r[8 * q + 7])
                         : "l"(p + 8 * q) : "memory");
    }
}

// ------------------------------------------------------- genetic value
// A warp's staged records: lane l = 4g + q holds row 8q + g, at position
// 8q + (g + 2q) % 8 of each 16-byte plane, so both the lanes' stores (any
// eight consecutive lanes) and ldmatrix (the eight rows of a matrix) touch
// all banks once.
__device__ __forceinline__ uint32_t stage_row(uint32_t lane) {
    const uint32_t g = lane >> 2, q = lane & 3u;
    return 16u * (8u * q + ((g + 2u * q) & 7u));
}
__device__ __forceinline__ uint32_t matrix_row(uint32_t lane) {  // ldmatrix: the row lane supplies the address of
    const uint32_t i = lane & 7u, q = lane >> 3;
    return 16u * (8u * q + ((i + 2u * q) & 7u));
}

template <int W>
__device__ __forceinline__ void stage_record(uint32_t addr, const uint32_t (&c)[2 * W]) {
    if constexpr (W == 1) {  // twice: every lane of a row's four finds one haplotype
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %1, %2};" ::"r"(addr), "r"(c[0]), "r"(c[1]) : "memory");
    } else {
#pragma unroll
        for (int p = 0; p < W / 2; ++p)
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr + 512u * p), "r"(c[4 * p]),
                         "r"(c[4 * p + 1]), "r"(c[4 * p + 2]), "r"(c[4 * p + 3]) : "memory");
    }
}
template <int W>
__device__ __forceinline__ void unstage_record(uint32_t addr, uint32_t (&c)[2 * W]) {
    if constexpr (W == 1) {
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(c[0]), "=r"(c[1]) : "r"(addr) : "memory");
    } else {
#pragma unroll
        for (int p = 0; p < W / 2; ++p)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(c[4 * p]), "=r"(c[4 * p + 1]), "=r"(c[4 * p + 2]), "=r"(c[4 * p + 3])
                         : "r"(addr + 512u * p) : "memory");
    }
}

// Words of a plane in fragment order: x[i] is word q of row 8i + g.
__device__ __forceinline__ void load_plane(uint32_t addr, uint32_t (&x)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(addr) : "memory");
}

__device__ __forceinline__ void mma_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// N element pairs of every row (x: the four rows' words) from bit positions
// 0, STEP, 2 STEP, ... of both half words times their fragments.  Positions
// past the linear range come down by shifting the word (STEP 2: the seventh
// and eighth by 4, STEP 1: from the twelfth on by 5).
template <int N, int STEP>
__device__ __forceinline__ void add_elements(float (&c0)[4], float (&c1)[4], const uint32_t (&x)[4], uint32_t frag) {
    constexpr int LIN = STEP == 2 ? 6 : 11, SHIFT = STEP == 2 ? 4 : 5;
    constexpr uint32_t ONE = STEP == 2 ? 0x00030003u : 0x00010001u;
    uint32_t b[4];
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        if (i % 4 == 0)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(frag + 128u * i) : "memory");
        uint32_t e[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = i + h;
#pragma unroll
            for (int r = 0; r < 4; ++r)
                e[h][r] = (k < LIN ? x[r] : x[r] >> SHIFT) & (ONE << (k < LIN ? STEP * k : STEP * k - SHIFT));
        }
        mma_f16(c0, e[0][0], e[0][1], e[1][0], e[1][1], b[i % 4], b[i % 4 + 1]);
        mma_f16(c1, e[0][2], e[0][3], e[1][2], e[1][3], b[i % 4], b[i % 4 + 1]);
    }
}

// Genetic value and allele count of the lane's own staged record.  frag: the
// shared address of the value fragments.
template <int W, class SM>
__device__ __forceinline__ void staged_value(uint32_t planes, uint32_t lane, uint32_t frag, bool dom, bool two_digits,
                                             int32_t &raw, uint32_t &allele) {
    const uint32_t at = planes + matrix_row(lane);
    const uint32_t sh = W >= 4 ? 0u : W == 2 ? 8u * ((lane >> 1) & 1u) : 4u * (lane & 3u);  // the lane's part of a word
    float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int s = 0; s < (int)SM::kSets; ++s) {
        uint32_t x[4], y[4];
        load_plane(at + 512u * s, x);
        if constexpr (W <= 2) {  // the other haplotype's word sits in the lane W away
#pragma unroll
            for (int i = 0; i < 4; ++i) y[i] = __shfl_xor_sync(0xFFFFFFFFu, x[i], W);
        } else {
            load_plane(at + 512u * (s + (int)SM::kSets), y);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // x: heterozygous loci, y: homozygous for allele 1
            const uint32_t t = x[i] ^ y[i];
            y[i] &= x[i];
            x[i] = t;
        }
        const uint32_t f0 = frag + s * SM::kSetBytes + 16u * lane;
        if (!dom) {
            constexpr uint32_t EVEN = 0x55555555u;
            constexpr int N = (int)SM::kRegs / 2;
            uint32_t z[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) z[i] = ((x[i] & EVEN) | ((y[i] << 1) & ~EVEN)) >> sh;
            add_elements<N, 2>(c0, c1, z, f0);
#pragma unroll
            for (int i = 0; i < 4; ++i) z[i] = (((x[i] >> 1) & EVEN) | (y[i] & ~EVEN)) >> sh;
            add_elements<N, 2>(c0, c1, z, f0 + SM::kSetBytes / 2u);
        } else {
            if constexpr (W < 4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    x[i] >>= sh;
                    y[i] >>= sh;
                }
            }
            add_elements<(int)SM::kRegs, 1>(c0, c1, x, f0);
            add_elements<(int)SM::kRegs, 1>(c0, c1, y, f0 + SM::kTabBytes);
        }
    }
    // this lane's row: 8q + g is row g or g + 8 of tile q / 2
    const bool up = (lane & 1u) != 0u, second = (lane & 2u) != 0u;
    const float lo = second ? (up ? c1[2] : c1[0]) : (up ? c0[2] : c0[0]);
    const float hi = second ? (up ? c1[3] : c1[1]) : (up ? c0[3] : c0[1]);
    // a sum * 2^20 is a whole number below 2^22: read it off the mantissa
    constexpr float kScale = 1048576.f, kMagic = 12582912.f;
    raw = __float_as_int(fmaf(lo, kScale, kMagic)) - 0x4B400000;
    const int32_t odd = __float_as_int(fmaf(hi, kScale, kMagic)) - 0x4B400000;
    allele = (uint32_t)odd;
    if (two_digits) raw += odd * 2048;
}

// Flip K distinct uniformly drawn positions of the lane's staged record
// (per-locus mutation; the draws of mutate()).  Rare, so kept out of line: it
// would cost every offspring the registers of its bookkeeping.
__device__ __noinline__ void mutate_staged(uint32_t row, uint32_t copies, uint32_t k, uint32_t j, uint32_t g,
                                           uint32_t rep, uint32_t k0, uint32_t k1) {
    uint16_t taken[kMaxKmax];
    uint32_t chosen = 0;
    k = min(k, (uint32_t)kMaxKmax);
    for (uint32_t a4 = 0; a4 < kMutDraws / 4 && chosen < k; ++a4) {
        const uint4 d = philox(make_uint4(j, g, rep, (kMutPos << 24) | a4), k0, k1);
        for (int l = 0; l < 4 && chosen < k; ++l) {
            const uint32_t pos = __umulhi(lane_of(d, l), copies);  // [0, 2L)
            bool dup = false;
            for (uint32_t i = 0; i < chosen; ++i) dup |= taken[i] == pos;
            if (!dup) {
                taken[chosen++] = (uint16_t)pos;
                const uint32_t w = pos >> 5, at = row + 512u * (w >> 2) + 4u * (w & 3u);
                uint32_t v;
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
                asm volatile("st.shared.u32 [%0], %1;" ::"r"(at), "r"(v ^ (1u << (pos & 31u))) : "memory");
            }
        }
    }
}

// ------------------------------------------------------- Philox
// Philox4x32-10 (see device_common.cuh) at counters (j, g, rep, word): the
// round keys come from the kernel's parameters, and what the first two rounds
// share is made once -- A * j per offspring, the rest (g, rep) per generation.
struct GenRng {
    uint32_t hx, lx, cy;  // product of A and word 0 after round 0 (hx with round 1's key), word 1 with round 1's key
};
using RoundKeys = uint32_t[20];
constexpr uint32_t kPhA = 0xD2511F53u, kPhB = 0xCD9E8D57u;
__device__ __forceinline__ GenRng gen_rng(const RoundKeys &keys, uint32_t rep, uint32_t g) {
    const unsigned long long q = (unsigned long long)kPhB * rep;
    const unsigned long long p = (unsigned long long)kPhA * ((uint32_t)(q >> 32) ^ g ^ keys[0]);
    return GenRng{(uint32_t)(p >> 32) ^ keys[3], (uint32_t)p, (uint32_t)q ^ keys[2]};
}
__device__ __forceinline__ uint4 philox_at(const RoundKeys &keys, const GenRng &r, unsigned long long aj, uint32_t word) {
    unsigned long long p1 = (unsigned long long)kPhB * ((uint32_t)(aj >> 32) ^ word ^ keys[1]), p0;
    uint4 c = make_uint4((uint32_t)(p1 >> 32) ^ r.cy, (uint32_t)p1, r.hx ^ (uint32_t)aj, r.lx);
#pragma unroll
    for (int i = 2; i < 10; ++i) {
        p0 = (unsigned long long)kPhA * c.x;
        p1 = (unsigned long long)kPhB * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ keys[2 * i], (uint32_t)p1,
                       (uint32_t)(p0 >> 32) ^ c.w ^ keys[2 * i + 1], (uint32_t)p0);
    }
    return c;
}

// ------------------------------------------------------- linkage map
// A linkage map in shared memory (see LinkParams).
struct LinkMap {
    const uint32_t *cdf, *cum, *guide;
    const uint16_t *first;  // first locus of each chromosome, 0xFFFF past the last
    uint32_t kmax;
    uint32_t *tog;          // the warp's toggle words [gamete][W][lane]
};

// Origin masks of both gametes of a warp's 32 offspring under the linkage map
// (bit set: the locus comes from the parent's haplotype 1); all lanes take
// part, valid = false gives a lane no crossovers.  A crossover toggles its
// first locus; a prefix XOR over the whole genome turns the toggles into
// flips, and a chromosome's flips are brought to its coin at its first locus
// by one comparison with the bit before it, so neither a crossover's
// chromosome nor its end has to be found (applying each chromosome's coin and
// end toggles took a quarter of the kernel).  The crossovers are dealt to the
// warp's lanes one Philox block (up to four crossovers of one gamete) at a
// time instead of each lane looping over its own, which would run the warp to
// its lanes' largest count; toggles go to the owner's words in shared memory
// by atomic XOR.
template <int W>
__device__ __forceinline__ void linked_masks(const LinkMap &lk, const RoundKeys &keys, const GenRng &rng, uint32_t j,
                                             bool valid, uint32_t (&mm)[W], uint32_t (&mf)[W]) {
    constexpr uint32_t L = 32u * W;
    const uint32_t lane = threadIdx.x & 31u;
    const unsigned long long aj = (unsigned long long)kPhA * j;
    uint4 d0[2];
    uint32_t K[2];
#pragma unroll
    for (uint32_t pi = 0; pi < 2u; ++pi) {
        d0[pi] = philox_at(keys, rng, aj, (kLink << 24) | (pi << 8));
        uint32_t k = 0;
        if (valid && lk.kmax != 0u && d0[pi].x >= lk.cdf[0]) {
            k = 1u;
#pragma unroll
            for (uint32_t step = 16u; step > 0u; step >>= 1)
                if (k + step <= lk.kmax && lk.cdf[k + step - 1u] <= d0[pi].x) k += step;
        }
        K[pi] = k;
#pragma unroll
        for (uint32_t w = 0; w < (uint32_t)W; ++w) lk.tog[(pi * W + w) * 32u + lane] = 0u;
    }
    // this lane's Philox blocks of crossovers, both gametes, and the warp's offsets
    const uint32_t nb0 = (K[0] + 3u) >> 2, nb = nb0 + ((K[1] + 3u) >> 2);
    uint32_t off = nb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, off, o);
        if ((int)lane >= o) off += y;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, off, 31);
    off -= nb;  // exclusive
    const uint32_t mine = off | nb0 << 10 | K[0] << 14 | K[1] << 20;  // off <= 512, nb0 <= 8, K <= 32
    __syncwarp();
    for (uint32_t f0 = 0; f0 < total; f0 += 32u) {
        const uint32_t f = f0 + lane;
        uint32_t o = 0;  // the owner: the last lane whose offset is <= f
#pragma unroll
        for (uint32_t step = 16u; step > 0u; step >>= 1) {
            const uint32_t v = __shfl_sync(0xFFFFFFFFu, off, (int)(o + step));
            if (v <= f) o += step;
        }
        const uint32_t x = __shfl_sync(0xFFFFFFFFu, mine, (int)o), oj = __shfl_sync(0xFFFFFFFFu, j, (int)o);
        if (f < total) {
            const uint32_t onb0 = (x >> 10) & 15u, b = f - (x & 1023u), pi = b < onb0 ? 0u : 1u,
                           blk = pi ? b - onb0 : b, Kp = pi ? x >> 20 : (x >> 14) & 63u;
            const uint4 d = philox_at(keys, rng, (unsigned long long)kPhA * oj, (kLink << 24) | (pi << 8) | (1u + blk));
            uint32_t *ot = lk.tog + pi * W * 32u + o;
#pragma unroll
            for (uint32_t l = 0; l < 4u; ++l) {
                if (4u * blk + l < Kp) {
                    const uint32_t u = lane_of(d, (int)l);
                    const uint32_t ge = lk.guide[u >> (32 - kLinkGuideBits)], nbd = ge >> 26;
                    uint32_t I = ge & 0xFFu;  // the bucket's first interval; with no boundary in it, cum[I] > u
                    I = min(I + (lk.cum[I] <= u ? 1u : 0u), L - 1u);
                    if (nbd > 1u)
                        while (I + 1u < L && lk.cum[I] <= u) ++I;
                    atomicXor(ot + (I >> 5) * 32u, 1u << (I & 31u));
                }
            }
        }
    }
    __syncwarp();
    uint32_t before[2] = {0u, 0u};  // the flip of the locus before the word
    uint32_t fix[2] = {0u, 0u};     // all ones where the running chromosome's flips are inverted
    uint32_t coins[2][3] = {{d0[0].y, d0[0].z, d0[0].w}, {d0[1].y, d0[1].z, d0[1].w}};  // the next chromosome's lowest
    uint32_t c = 0, next = 0u;      // the next chromosome and its first locus
#pragma unroll
    for (uint32_t w = 0; w < (uint32_t)W; ++w) {
        uint32_t x[2], shifted[2], F[2];
#pragma unroll
        for (uint32_t pi = 0; pi < 2u; ++pi) {
            uint32_t y = lk.tog[(pi * W + w) * 32u + lane];
            y ^= y << 1;
            y ^= y << 2;
            y ^= y << 4;
            y ^= y << 8;
            y ^= y << 16;
            x[pi] = y ^ (0u - before[pi]);
            shifted[pi] = x[pi] << 1 | before[pi];  // the flip before each locus
            before[pi] = x[pi] >> 31;
            F[pi] = fix[pi];
        }
        while (next < 32u * (w + 1u)) {  // chromosomes that start in this word (the same in all lanes)
            const uint32_t s = next & 31u, from = 0xFFFFFFFFu << s;
#pragma unroll
            for (uint32_t pi = 0; pi < 2u; ++pi) {
                fix[pi] = 0u - ((coins[pi][0] ^ (shifted[pi] >> s)) & 1u);
                F[pi] = (F[pi] & ~from) | (fix[pi] & from);
                coins[pi][0] = __funnelshift_r(coins[pi][0], coins[pi][1], 1);
                coins[pi][1] = __funnelshift_r(coins[pi][1], coins[pi][2], 1);
                coins[pi][2] >>= 1;
            }
            next = lk.first[++c];
        }
        mm[w] = x[0] ^ F[0];
        mf[w] = x[1] ^ F[1];
    }
}

// ------------------------------------------------------- parents
// Records of the survivors drawn by u0 and u1 (rank u * S / 2^32) in the slot
// layout.  one_step: no guide entry is more than one slot behind
// (build_directory), so the search is a select.
template <class SM>
__device__ __forceinline__ void locate(const SoloArgs &a, uint32_t u0, uint32_t u1, uint32_t S, bool one_step,
                                       uint32_t &i0, uint32_t &i1) {
    auto guide = [&](uint32_t u) {
        return (uint32_t)*reinterpret_cast<const uint16_t *>(g_smem + SM::kGuideOff + 2u * (u >> (32u - a.guide_bits)));
    };
    auto slot = [&](uint32_t s) { return *reinterpret_cast<const uint2 *>(g_smem + SM::kDir + 8u * s); };
    const uint32_t r0 = __umulhi(u0, S), r1 = __umulhi(u1, S);
    uint32_t s0 = guide(u0), s1 = guide(u1);
    uint2 e0 = slot(s0), e1 = slot(s1);
    if (one_step) {
        const uint32_t rec = a.slot_len * 32u;
        i0 = r0 < e0.x ? r0 + e0.y : r0 - e0.x + (s0 + 1u) * rec;
        i1 = r1 < e1.x ? r1 + e1.y : r1 - e1.x + (s1 + 1u) * rec;
        return;
    }
    while (e0.x <= r0) e0 = slot(++s0);  // the last slot's end is S > r
    while (e1.x <= r1) e1 = slot(++s1);
    i0 = r0 + e0.y;
    i1 = r1 + e1.y;
}

// Weighted parents (bounded rejection): proposals in
// pairs, both roles together; thr holds each survivor's thresholds as mother
// and as father at its record's place.
template <class SM>
__device__ __forceinline__ void weighted_records(const SoloArgs &a, const RoundKeys &keys, const uint2 *thr, const GenRng &rng,
                                                 unsigned long long aj, uint32_t S, bool one_step,
                                                 uint32_t &mom,
                                                 uint32_t &dad) {
    bool open_m = true, open_f = true;
    for (uint32_t k = 0; k < kMateAttempts && (open_m || open_f); k += 2) {
        const uint32_t sub = (kMateW << 24) | (k >> 1);
        uint4 dm = make_uint4(0u, 0u, 0u, 0u), df = dm;
        uint32_t rm0 = 0, rm1 = 0, rf0 = 0, rf1 = 0, tm0 = 0, tm1 = 0, tf0 = 0, tf1 = 0;
        if (open_m) {
            dm = philox_at(keys, rng, aj, sub);
            locate<SM>(a, dm.x, dm.z, S, one_step, rm0, rm1);
            tm0 = __ldcg(&thr[rm0].x);
            tm1 = __ldcg(&thr[rm1].x);
        }
        if (open_f) {
            df = philox_at(keys, rng, aj, sub | (1u << 8));
            locate<SM>(a, df.x, df.z, S, one_step, rf0, rf1);
            tf0 = __ldcg(&thr[rf0].y);
            tf1 = __ldcg(&thr[rf1].y);
        }
        if (open_m) {
            const bool a0 = tm0 == kCertain || dm.y < tm0, a1 = tm1 == kCertain || dm.w < tm1;
            mom = a0 ? rm0 : rm1;
            open_m = !(a0 || a1);
        }
        if (open_f) {
            const bool a0 = tf0 == kCertain || df.y < tf0, a1 = tf1 == kCertain || df.w < tf1;
            dad = a0 ? rf0 : rf1;
            open_f = !(a0 || a1);
        }
    }
}

// ------------------------------------------------------- the directory
// Exclusive scan of the slots' survivor counts into the block's directory and
// guide, by all warps but the block's last (which has the resource to close).
// Slot s holds ranks P[s] .. P[s+1]-1; entry s is {P[s+1], s * slot_records -
// P[s]}.  Guide entry h is a slot at or just before the one of the smallest
// rank drawn by a u whose top bits are h, rank floor(h S / entries): slot s
// enters the guide at the first h surely past entries * P[s] / S.  Every block
// does this every generation, so it takes a handful of instructions a slot
// (exact entries by 64-bit products took a sixth of a generation at N = 10^6)
// and the guide grows with the slots (four to eight entries each, 3.4 at the
// most slots).  Writes the total to *total; with no survivors the tables stay
// as they are.  Returns whether every slot of the thread holds more ranks than
// two guide entries span, so that a rank lies in its entry's slot or the next.
// PER: runs of 32 slots a warp takes, at most; OWN: with one run, the count of
// the thread's slot is `own` already.
template <class SM, uint32_t PER, bool OWN>
__device__ __forceinline__ bool directory_of(const uint32_t *counts, uint32_t first, uint32_t nslots, uint32_t slot_records,
                                                uint32_t guide_bits, uint32_t *s_warp, uint32_t *total) {
    constexpr uint32_t T = SM::kThreads - 32u, NW = T / 32u;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    // warp w takes per runs of 32 consecutive slots from s0, lane l slot l of each
    const uint32_t per = (nslots + T - 1) / T, s0 = warp * 32u * per + lane;
    uint32_t c[PER], own = 0;
#pragma unroll
    for (uint32_t i = 0; i < PER; ++i) {
        c[i] = i < per && s0 + 32u * i < nslots ? OWN && PER == 1u ? first : __ldcg(counts + s0 + 32u * i) : 0u;
        own += c[i];
    }
    own = __reduce_add_sync(0xFFFFFFFFu, own);
    if (lane == 0u) s_warp[warp] = own;
    asm volatile("bar.sync 1, %0;" ::"n"(T) : "memory");
    const uint32_t w = lane < NW ? s_warp[lane] : 0u;
    const uint32_t S = __reduce_add_sync(0xFFFFFFFFu, w);
    if (tid == 0u) *total = S;
    if (S == 0u) return true;
    uint32_t P = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? w : 0u);
    // the first h with floor(h S / entries) >= P, or one later when the float
    // quotient (off by less than 0.004) is too close to tell
    const uint32_t entries = 1u << guide_bits, span = 2u * (S >> guide_bits) + 2u;
    const float inv = (float)entries / (float)S;
    auto entry_of = [&](uint32_t p) { return p ? min((uint32_t)fmaf((float)p, inv, 1.005f), entries) : 0u; };
    // all runs stage by stage, so that their latencies overlap
    uint32_t end[PER], h[PER];
#pragma unroll
    for (uint32_t i = 0; i < PER; ++i) end[i] = c[i];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (uint32_t i = 0; i < PER; ++i) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, end[i], o);
            if ((int)lane >= o) end[i] += y;
        }
    bool wide = true;
    uint32_t run = entry_of(P), left = 0;  // the run's first guide entry, the most entries a slot has
#pragma unroll
    for (uint32_t i = 0; i < PER; ++i) {
        const uint32_t s = s0 + 32u * i;
        end[i] += P;
        P = __shfl_sync(0xFFFFFFFFu, end[i], 31);
        const bool mine = i < per && s < nslots;
        if (mine)
            *reinterpret_cast<uint2 *>(g_smem + SM::kDir + 8u * s) = make_uint2(end[i], s * slot_records - (end[i] - c[i]));
        wide = wide && (c[i] > span || !mine);
        end[i] = entry_of(end[i]);  // from here on the slot's last entry
        const uint32_t before = __shfl_up_sync(0xFFFFFFFFu, end[i], 1);
        h[i] = lane ? before : run;
        run = __shfl_sync(0xFFFFFFFFu, end[i], 31);
        left = max(left, end[i] - h[i]);
    }
    for (uint32_t k = 0; k < left; ++k) {
#pragma unroll
        for (uint32_t i = 0; i < PER; ++i)
            if (h[i] + k < end[i])
                *reinterpret_cast<uint16_t *>(g_smem + SM::kGuideOff + 2u * (h[i] + k)) = (uint16_t)(s0 + 32u * i);
    }
    return wide;
}
// (Two runs a warp have an instance but at L = 256: as six, calls of one generation
// of N = 20,000 x 32 took 11.4 us instead of 10.1; at L = 256 the instance cost the
// kernel one percent at every size.)
template <class SM, bool OWN>
__device__ __forceinline__ bool build_directory(const uint32_t *counts, uint32_t own, uint32_t nslots, uint32_t slot_records,
                                                uint32_t guide_bits, uint32_t *s_warp, uint32_t *total) {
    constexpr uint32_t T = SM::kThreads - 32u;
    if (nslots <= T) return directory_of<SM, 1, OWN>(counts, own, nslots, slot_records, guide_bits, s_warp, total);
    if (SM::kPlanes < 4u && nslots <= 2u * T) return directory_of<SM, 2, OWN>(counts, own, nslots, slot_records, guide_bits, s_warp, total);
    return directory_of<SM, (SM::kSlots + T - 1) / T, OWN>(counts, own, nslots, slot_records, guide_bits, s_warp, total);
}

// ------------------------------------------------------- per-locus counts
// Allele copies of the block's own records [j0, j1), added to the generation's
// row: bit-sliced counters per lane (plane k holds bit k of every locus's count
// among the lane's records), transposed across the warp before they could
// overflow.  Four record words at a time.
__device__ __forceinline__ uint32_t transpose32(uint32_t x, uint32_t lane) {
    constexpr uint32_t M[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const uint32_t s = 16u >> k;
        const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, (int)s);
        x = (lane & s) ? (((y >> s) & M[k]) | (x & ~M[k])) : ((x & M[k]) | ((y << s) & ~M[k]));
    }
    return x;
}
template <int W, int BLOCK>
__device__ __forceinline__ void count_loci(const uint32_t *geno, uint32_t j0, uint32_t j1, uint32_t *s_cnt,
                                           uint32_t *row) {
    constexpr uint32_t L = 32u * W, NW = BLOCK / 32;
    constexpr int C = W == 1 ? 2 : 4, K = kLocusPlanes;  // words of one pass
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    for (uint32_t i = tid; i < L; i += BLOCK) s_cnt[i] = 0u;
    __syncthreads();  // and the block's records are written
#pragma unroll 1
    for (int p = 0; p < 2 * W / C; ++p) {
        uint32_t v[C][K], held = 0;
#pragma unroll
        for (int c = 0; c < C; ++c)
#pragma unroll
            for (int k = 0; k < K; ++k) v[c][k] = 0u;
        auto flush = [&]() {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                uint32_t sum = 0;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    sum += (uint32_t)__popc(transpose32(v[c][k], lane)) << k;
                    v[c][k] = 0u;
                }
                atomicAdd(&s_cnt[32u * (uint32_t)((p * C + c) % W) + lane], sum);
            }
            held = 0;
        };
        for (uint32_t j = j0 + 32u * warp; j < j1; j += 32u * NW) {
            uint32_t x[C];
            const uint32_t *src = geno + (size_t)(j + lane) * (2 * W) + C * p;
            if (j + lane < j1) {
                if constexpr (C == 2) {
                    const uint2 u = __ldcg(reinterpret_cast<const uint2 *>(src));
                    x[0] = u.x;
                    x[1] = u.y;
                } else {
                    const uint4 u = __ldcg(reinterpret_cast<const uint4 *>(src));
                    x[0] = u.x;
                    x[1] = u.y;
                    x[2] = u.z;
                    x[3] = u.w;
                }
            } else {
#pragma unroll
                for (int c = 0; c < C; ++c) x[c] = 0u;
            }
#pragma unroll
            for (int c = 0; c < C; ++c) {  // ripple-carry add of one bit per locus
                uint32_t carry = x[c];
#pragma unroll
                for (int k = 0; k < K - 1; ++k) {
                    const uint32_t t = v[c][k] & carry;
                    v[c][k] ^= carry;
                    carry = t;
                }
                v[c][K - 1] ^= carry;
            }
            if (++held == (1u << K) - 1u) flush();
        }
        if (held) flush();
    }
    __syncthreads();
    for (uint32_t i = tid; i < L; i += BLOCK)
        if (s_cnt[i]) atomicAdd(row + i, s_cnt[i]);
}

// ------------------------------------------------------- the kernel
// A lane's statistics of one generation, and their exact sums over the block:
// every lane leaves its own in shared memory, and after a block barrier warp k
// takes field k (a reduction in every warp took three times as long).
struct LaneStats {
    long long sum_raw = 0, sum_raw_s = 0;
    unsigned long long sum_raw2 = 0, cons = 0;
    uint32_t het = 0, allele = 0;
    int mn = INT_MAX, mx = INT_MIN;
};
template <class SM>
__device__ __forceinline__ void put_stats(const LaneStats &ts, uint32_t tid) {
    unsigned long long *s64 = reinterpret_cast<unsigned long long *>(g_smem + SM::kStats) + tid;
    s64[0] = (unsigned long long)ts.sum_raw;
    s64[SM::kThreads] = (unsigned long long)ts.sum_raw_s;
    s64[2 * SM::kThreads] = ts.sum_raw2;
    s64[3 * SM::kThreads] = ts.cons;
    uint32_t *s32 = reinterpret_cast<uint32_t *>(g_smem + SM::kStats + 32u * SM::kThreads) + tid;
    s32[0] = ts.het;
    s32[SM::kThreads] = ts.allele;
    s32[2 * SM::kThreads] = (uint32_t)ts.mn;
    s32[3 * SM::kThreads] = (uint32_t)ts.mx;
}
template <class SM>
__device__ __forceinline__ void add_stats(GenAcc *acc, uint32_t warp, uint32_t lane) {
    if (warp >= 8u) return;
    if (warp < 6u) {
        unsigned long long x = 0;
#pragma unroll
        for (uint32_t i = 0; i < SM::NW; ++i)
            x += warp < 4u ? *reinterpret_cast<const unsigned long long *>(g_smem + SM::kStats +
                                                                           8u * (warp * SM::kThreads + 32u * i + lane))
                           : sm_u32(SM::kStats + 32u * SM::kThreads + 4u * ((warp - 4u) * SM::kThreads + 32u * i + lane));
        x = warp_sum_u64(x);  // modulo 2^64: signed sums too
        if (lane == 0u) atomicAdd(&acc->sum[warp], x);
    } else {
        int x = warp == 6u ? INT_MAX : INT_MIN;
#pragma unroll
        for (uint32_t i = 0; i < SM::NW; ++i) {
            const int y = (int)sm_u32(SM::kStats + 32u * SM::kThreads + 4u * ((warp - 4u) * SM::kThreads + 32u * i + lane));
            x = warp == 6u ? min(x, y) : max(x, y);
        }
        x = warp == 6u ? __reduce_min_sync(0xFFFFFFFFu, x) : __reduce_max_sync(0xFFFFFFFFu, x);
        if (lane == 0u) {
            if (warp == 6u) atomicMin(&acc->mn, x);
            else atomicMax(&acc->mx, x);
        }
    }
}

// GENERAL: dominance, values beyond 2048 in magnitude or a bias beyond 2^30
// (the others' instance has none of these branches in its loop).
// Blocks 0 .. team - 1 (this one is `rank`) form n_gen generations of a
// population; keep_last: the last of them is the call's last; single: one
// generation, closed by the kernel launched next (k_close).
template <int W, bool LINKED, bool WEIGHTED, bool GENERAL>
__device__ __forceinline__ void form_generations(const SoloArgs &a, const RoundKeys &keys, uint32_t n_gen,
                                                 bool keep_last, bool single, uint32_t rank, uint32_t team) {
    constexpr int BLOCK = (int)kSoloThreads;
    using SM = GenSmem<W, LINKED>;
    constexpr uint32_t NW = BLOCK / 32;
    __shared__ uint32_t s_cdf[kMaxKmax];
    __shared__ uint32_t s_scan[32];
    __shared__ uint32_t s_cnt[32 * W];
    __shared__ uint32_t s_total, s_f[2], s_now[8];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(g_smem);
    const PopParams *P = a.prm;
    DevState *st = a.state;

    // tables
    const bool eco = a.has_eco != 0u, dom = GENERAL && a.dom != 0u;
    for (uint32_t i = tid; i < (uint32_t)kBins / 4u; i += BLOCK) {
        cp_async_16(smem0 + SM::kThr + 16u * i, P->table + 4u * i);
        if (eco) cp_async_16(smem0 + SM::kAtt + 16u * i, P->attack + 4u * i);
    }
    for (uint32_t i = tid; i < SM::kTabBytes / 16u; i += BLOCK) {
        cp_async_16(smem0 + SM::kFrag + 16u * i, a.frag->table[0] + 4u * i);
        if (dom) cp_async_16(smem0 + SM::kFrag + SM::kTabBytes + 16u * i, a.frag->table[1] + 4u * i);
    }
    cp_async_commit();
    if (tid < (uint32_t)kMaxKmax) s_cdf[tid] = tid < a.kmax ? P->cdf[tid] : 0xFFFFFFFFu;
    LinkMap lk{};
    if constexpr (LINKED) {
        const LinkParams *lp = P->link;
        uint32_t *cdf = reinterpret_cast<uint32_t *>(g_smem + SM::kLinkOff), *cum = cdf + kMaxKmax, *gd = cum + kMaxLoci;
        uint16_t *first = reinterpret_cast<uint16_t *>(gd + kLinkGuide);
        if (tid < (uint32_t)kMaxKmax) cdf[tid] = lp->cdf[tid];
        for (uint32_t i = tid; i < 32u * W; i += BLOCK) cum[i] = lp->cum[i];
        for (uint32_t i = tid; i < (uint32_t)kLinkGuide; i += BLOCK) gd[i] = lp->guide[i];
        if (tid <= (uint32_t)kMaxChrom) first[tid] = tid < lp->nchrom ? lp->first[tid] : (uint16_t)0xFFFFu;
        lk = LinkMap{cdf, cum, gd, first, lp->kmax,
                     reinterpret_cast<uint32_t *>(g_smem + SM::kStage + warp * SM::kPerWarp)};
    }
    griddep_wait();  // the tables are parameters: nothing an earlier launch writes
    griddep_release();
    // the call's starting state (written by earlier launches): read once for the
    // block -- by every thread, it kept one line of L2 busy for microseconds, and a
    // teammate that gives up on a block this late may change the status meanwhile
    static_assert(offsetof(DevState, S) == 4 && offsetof(DevState, f) == 8 && offsetof(DevState, status) == 12 &&
                      offsetof(DevState, R) == 16 && offsetof(DevState, target) == 28,
                  "the state's first eight words");
    if (tid < 8u && tid != 6u) s_now[tid] = ld_relaxed_u32(reinterpret_cast<const uint32_t *>(st) + tid);
    // survivors of the thread's first slot, of both parities, so that the load
    // does not wait for the state
    const uint32_t own0 = tid < a.nslots ? __ldcg(a.counts[0] + tid) : 0u,
                   own1 = tid < a.nslots ? __ldcg(a.counts[1] + tid) : 0u;
    __syncthreads();
    uint32_t gen = s_now[0], f = s_now[2];
    const uint32_t target = s_now[7];
    double R = __hiloint2double((int)s_now[5], (int)s_now[4]);
    const bool over = (int32_t)s_now[3] != SPG_OK || s_now[1] == 0u || gen >= target;
    if (single && rank == 0u && tid == 0u) st->done = over ? 0u : gen + 1u;  // the generation to be closed
    if (over) {
        cp_async_wait<0>();
        return;
    }

    const uint32_t rep = a.rep, k0 = keys[0], k1 = keys[1];
    const uint32_t rec_slot = a.slot_len * 32u;
    const uint32_t stage = smem0 + SM::kStage + warp * SM::kPerWarp, my_row = stage + stage_row(lane);
    const uint32_t slot0 = (uint32_t)(((unsigned long long)a.nslots * rank) / team);
    const uint32_t slot1 = (uint32_t)(((unsigned long long)a.nslots * (rank + 1u)) / team);
    bool one_step = true;
    if (warp + 1u < NW)
        one_step = build_directory<SM, true>(a.counts[gen & 1u], (gen & 1u) ? own1 : own0, a.nslots, rec_slot,
                                             a.guide_bits, s_scan, &s_total);
    cp_async_wait<0>();  // the tables have landed meanwhile
    one_step = __syncthreads_and(one_step) != 0;
    uint32_t S = s_total;

    bool again = false;  // a generation without survivors formed once more for its full records
    for (uint32_t done = 0; done < n_gen && (gen < target || again);) {
        const uint32_t g = again ? gen : gen + 1u;
        const bool list = again || (keep_last && done + 1u == n_gen) || g == target;
        const bool full = list || a.locus_row[0] != nullptr;
        const uint32_t *par = a.packed[(g + 1u) & 1u];
        uint32_t *out = a.packed[g & 1u];
        const GenRng rng = gen_rng(keys, rep, g);
        double grown = 0.0;  // the resource before consumption (the block's last warp), while the generation is formed
        if (eco && tid == BLOCK - 32u)
            grown = a.eco_model == 1u
                        ? resource_grown_bh(R, growth_rate(a.eco_r, a.eco_r_sd, g, rep, k0, k1), a.eco_K)
                        : resource_grown(R, a.eco_r, a.eco_K);
        LaneStats ts;
        {
            // (A) a group's mate draw and parents; the next group's records are
            // on their way while a group is formed
            auto draw = [&](uint32_t j, uint4 &r, uint32_t (&pm)[2 * W], uint32_t (&pf)[2 * W]) {
                const unsigned long long aj = (unsigned long long)kPhA * j;
                r = philox_at(keys, rng, aj, kMate << 24);
                uint32_t mom, dad;
                if constexpr (WEIGHTED) {
                    weighted_records<SM>(a, keys, a.mate[(g + 1u) & 1u], rng, aj, S, one_step, mom, dad);
                } else {
                    locate<SM>(a, r.x, r.y, S, one_step, mom, dad);
                }
                load_packed<W>(par + (size_t)mom * (2 * W), pm);
                load_packed<W>(par + (size_t)dad * (2 * W), pf);
            };
            uint4 r_next;
            uint32_t pm_next[2 * W], pf_next[2 * W];
            // the warp's groups, slot after slot
            uint32_t slot = slot0 + warp, base = slot * rec_slot, end = min(base + rec_slot, a.n), at0 = base, j0 = base;
            if (slot < slot1) draw(base + lane, r_next, pm_next, pf_next);
#pragma unroll 1
            while (slot < slot1) {
                const uint32_t j = j0 + lane;
                const bool valid = j < a.n;
                const uint4 r = r_next;
                // (B) gametes: the mask streams, or the linkage map's masks
                uint32_t ch[2 * W];
                if constexpr (LINKED) {
                    uint32_t mm[W], mf[W];
                    linked_masks<W>(lk, keys, rng, j, valid, mm, mf);
                    __syncwarp();  // the toggles' memory holds the staged records next
#pragma unroll
                    for (int w = 0; w < W; ++w) {
                        ch[w] = (pm_next[w] & ~mm[w]) | (pm_next[W + w] & mm[w]);
                        ch[W + w] = (pf_next[w] & ~mf[w]) | (pf_next[W + w] & mf[w]);
                    }
                } else {
                    const unsigned long long aj = (unsigned long long)kPhA * j;
#pragma unroll
                    for (int q4 = 0; q4 < (2 * W + 3) / 4; ++q4) {
                        const uint4 d = philox_at(keys, rng, aj, (kRecomb << 24) | (uint32_t)q4);
                        const int w = 2 * q4;
                        ch[w] = (pm_next[w] & ~d.x) | (pm_next[W + w] & d.x);
                        ch[W + w] = (pf_next[w] & ~d.y) | (pf_next[W + w] & d.y);
                        if constexpr (W > 1) {
                            ch[w + 1] = (pm_next[w + 1] & ~d.z) | (pm_next[W + w + 1] & d.z);
                            ch[W + w + 1] = (pf_next[w + 1] & ~d.w) | (pf_next[W + w + 1] & d.w);
                        }
                    }
                }
                const bool slot_done = j0 + 32u >= end;
                const uint32_t j0_next = slot_done ? (slot + NW) * rec_slot : j0 + 32u;
                if (!slot_done || slot + NW < slot1) draw(j0_next + lane, r_next, pm_next, pf_next);
                stage_record<W>(my_row, ch);
                if (r.w >= a.mut_from) {  // (B) mutations, on the staged record
                    uint32_t k = 0;
                    for (uint32_t i = 0; i < a.kmax; ++i) k += (r.w >= s_cdf[i]) ? 1u : 0u;
                    mutate_staged(my_row, 64u * W, k, j, g, rep, k0, k1);
                    unstage_record<W>(my_row, ch);
                    if constexpr (W == 1) stage_record<W>(my_row, ch);
                }
                __syncwarp();
                // (C) genetic value
                int32_t raw;
                uint32_t allele, het = 0;
                staged_value<W, SM>(stage, lane, smem0 + SM::kFrag, dom, GENERAL && a.two_digits != 0u, raw, allele);
#pragma unroll
                for (int w = 0; w < W; ++w) het += __popc(ch[w] ^ ch[W + w]);
                if (GENERAL && a.two_digits) {
                    allele = 0;
#pragma unroll
                    for (int w = 0; w < 2 * W; ++w) allele += __popc(ch[w]);
                }
                // (D) survival: the bin's threshold scaled by the resource factor
                uint32_t bin;
                if (!GENERAL || a.narrow_bias) {  // raw + bias stays inside 32 bits
                    bin = (uint32_t)min(max((raw + a.bias) >> a.shift, 0), kBins - 1);
                } else {
                    const long long v = (long long)raw + (long long)a.bias;
                    bin = v < 0 ? 0u : (uint32_t)min(v >> a.shift, (long long)(kBins - 1));
                }
                uint32_t thr = sm_u32(SM::kThr + bin * 4u);
                thr = f != kCertain ? __umulhi(thr, f) : thr;
                const bool alive = valid && min(r.z, kCertain - 1u) < thr;  // kCertain: whatever the draw
                const uint32_t bits = __ballot_sync(0xFFFFFFFFu, alive);
                // (E) the survivor's record at its place in the slot
                const uint32_t at = at0 + __popc(bits & ((1u << lane) - 1u));
                at0 += __popc(bits);
                if (alive) {
                    store_record<W>(out + (size_t)at * (2 * W), ch);
                    if constexpr (WEIGHTED) {
                        const WeightParams *wt = P->weights;
                        a.mate[g & 1u][at] = make_uint2(__ldg(&wt->acc[0][bin]), __ldg(&wt->acc[1][bin]));
                    }
                    ts.sum_raw_s += raw;
                    if (eco) ts.cons += sm_u32(SM::kAtt + bin * 4u);
                }
                if (valid) {
                    ts.het += het;
                    ts.allele += allele;
                    ts.sum_raw += raw;
                    ts.sum_raw2 += (unsigned long long)((long long)raw * (long long)raw);
                    ts.mn = min(ts.mn, raw);
                    ts.mx = max(ts.mx, raw);
                    if (full) store_record<W>(a.geno + (size_t)j * (2 * W), ch);
                }
                if (full && lane == 0u) a.alive[j0 >> 5] = bits;
                if (slot_done) {
                    if (lane == 0u && !again) a.counts[g & 1u][slot] = at0 - base;
                    slot += NW;
                    base = at0 = j0_next;
                    end = min(base + rec_slot, a.n);
                }
                j0 = j0_next;
            }
        }
        if (again) break;
        put_stats<SM>(ts, tid);
        if (a.locus_row[0])
            count_loci<W, BLOCK>(a.geno, min(slot0 * rec_slot, a.n),
                                 (uint32_t)min((unsigned long long)slot1 * rec_slot, (unsigned long long)a.n), s_cnt,
                                 a.locus_row[g & 1u]);
        __syncthreads();
        GenAcc *acc = a.acc + (size_t)(g % 3u) * kGenAccCopies;
        add_stats<SM>(acc + rank % kGenAccCopies, warp, lane);
        if (single) return;
        if (!team_barrier(a.barrier, rank, team, a.barrier_tries)) {  // the generation fails: every block gives up
            if (tid == 0u) atomicExch(reinterpret_cast<int *>(&st->status), SPG_ERR_TIMEOUT);
            return;
        }
        // close the generation: every block builds the directory while its last
        // warp finishes the resource and factor (the same arithmetic in each);
        // block 0's last warp writes the statistics record and the state
        bool wide = true;
        unsigned long long sum = 0;
        if (warp + 1u < NW) {
            wide = build_directory<SM, false>(a.counts[g & 1u], 0u, a.nslots, rec_slot, a.guide_bits, s_scan, &s_total);
        } else if (eco || rank == 0u) {
            sum = total_stats(__ldcg(reinterpret_cast<const unsigned long long *>(acc) + lane), lane);
            const unsigned long long cons = __shfl_sync(0xFFFFFFFFu, sum, 3);
            if (lane == 0u && eco) {
                R = resource_eaten(grown, cons);
                s_f[g & 1u] = factor_q32(R, a.eco_R_half);
            }
        }
        wide = __syncthreads_and(wide) != 0;
        const uint32_t S_new = s_total, f_new = eco ? s_f[g & 1u] : f;
        if (rank == 0u) {
            if (warp == NW - 1u) write_state(a, lane, g, sum, S_new, R, f_new);
            if (a.locus_row[0]) {  // the counted row to its place; clear for the generation after next
                uint32_t *row = a.locus_row[g & 1u], *dst = a.locus_ring + (size_t)((g - 1u) % a.locus_cap) * (32u * W);
                for (uint32_t i = tid; i < 32u * W; i += BLOCK) {
                    dst[i] = __ldcg(row + i);
                    row[i] = 0u;
                }
            }
        }
        if (list && S_new != 0u)
            list_survivors(a, 0u, a.nslots, rank * NW + warp, team * NW, lane, [] { return true; }, [&](uint32_t slot) {
                return slot * rec_slot - *reinterpret_cast<const uint32_t *>(g_smem + SM::kDir + 8u * slot + 4u);
            });
        gen = g;
        ++done;
        if (S_new == 0u) {
            if (list) break;  // its full records are written
            again = true;     // form it once more for them (its parents and directory are still there)
            --done;
            continue;
        }
        one_step = wide;
        S = S_new;
        f = f_new;
    }
}

// One population: every block of the grid is in its team.
template <int W, bool LINKED, bool WEIGHTED, bool GENERAL>
__global__ void __launch_bounds__(kSoloThreads, 1) k_generations(const __grid_constant__ SoloArgs a) {
    form_generations<W, LINKED, WEIGHTED, GENERAL>(a, a.keys, a.n_gen, a.keep_last != 0u, a.single != 0u,
                                                   blockIdx.x, gridDim.x);
}

// Several populations: each block works through its list of teams.  A team's
// blocks wait for one another, and all lists have the teams in one order, so
// the blocks of the first unfinished team are all at it or on their way.  A
// population stays with its team for the whole launch: its records stay in L2
// and no other population's generation waits for it.  Members of all locus
// counts share the launch (a launch per locus count left most blocks idle for
// batches of few members), the longest records first: a switch over the
// locus counts spilled in every body, one after the other they do not.  A
// member's arguments are in shared memory.
__shared__ SoloArgs s_team_args;
template <int W, bool LINKED, bool WEIGHTED, bool GENERAL>
__device__ __forceinline__ void team_places(const TeamArgs &t, uint32_t &p) {
    for (; p < t.block_places[blockIdx.x + 1u]; ++p) {
        const TeamPlace place = t.places[p];
        __syncthreads();  // the previous population's tables and arguments are no longer read
        for (uint32_t i = threadIdx.x; i < sizeof(SoloArgs) / 4u; i += kSoloThreads)
            reinterpret_cast<uint32_t *>(&s_team_args)[i] = reinterpret_cast<const uint32_t *>(t.members + place.member)[i];
        __syncthreads();
        if (s_team_args.words != (uint32_t)W) return;
        form_generations<W, LINKED, WEIGHTED, GENERAL>(s_team_args, s_team_args.keys, t.n_gen, t.keep_last != 0u,
                                                       t.single != 0u, place.rank, place.team);
    }
}
template <bool LINKED, bool WEIGHTED, bool GENERAL>
__global__ void __launch_bounds__(kSoloThreads, 1) k_teams(const __grid_constant__ TeamArgs t) {
    uint32_t p = t.block_places[blockIdx.x];
    team_places<8, LINKED, WEIGHTED, GENERAL>(t, p);
    team_places<4, LINKED, WEIGHTED, GENERAL>(t, p);
    team_places<2, LINKED, WEIGHTED, GENERAL>(t, p);
    team_places<1, LINKED, WEIGHTED, GENERAL>(t, p);
}

template <int W, bool LINKED, bool WEIGHTED>
SoloKernel solo_instance(bool general) {
    SoloKernel k;
    k.fn = general ? (const void *)&k_generations<W, LINKED, WEIGHTED, true>
                   : (const void *)&k_generations<W, LINKED, WEIGHTED, false>;
    k.smem = GenSmem<W, LINKED>::kBytes;
    return k;
}
template <bool LINKED, bool WEIGHTED, bool GENERAL>
SoloKernel team_instance() {
    SoloKernel k;
    k.fn = (const void *)&k_teams<LINKED, WEIGHTED, GENERAL>;
    k.smem = GenSmem<8, LINKED>::kBytes;  // the largest records' tables
    return k;
}

}  // namespace
}  // namespace spg
