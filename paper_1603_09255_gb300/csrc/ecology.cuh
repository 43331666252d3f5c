// The resource of a population's ecology (Fig. 1F): IEEE double with
// explicitly rounded basic operations, so that the oracle's host arithmetic
// agrees bit for bit.  Included by the kernels that close a generation.
#pragma once

#include "device_common.cuh"

namespace spg {
namespace {

// ------------------------------------------------------ ecology (Fig. 1F)
// The resource before consumption: logistic R + rR(1 - R/K), or the
// Beverton-Holt variant (r' R) / (1 + R/K).
__device__ double resource_grown(double R, double r, double K) {
    const double ratio = __ddiv_rn(R, K);
    const double room = __dsub_rn(1.0, ratio);
    const double rR = __dmul_rn(r, R);
    const double growth = __dmul_rn(rR, room);
    return __dadd_rn(R, growth);
}
__device__ double resource_grown_bh(double R, double rg, double K) {
    const double grown_num = __dmul_rn(rg, R);
    const double ratio = __ddiv_rn(R, K);
    const double den = __dadd_rn(1.0, ratio);
    return __ddiv_rn(grown_num, den);
}

// Less the consumption C 2^-16, clamped at 0.
__device__ double resource_eaten(double grown, unsigned long long C) {
    const double eaten = __dmul_rn(__ull2double_rn(C), 1.0 / 65536.0);
    double next = __dsub_rn(grown, eaten);
    if (!(next > 0.0)) next = 0.0;
    return next;
}

// Growth rate of generation g: r + r_sd * z, z the Irwin-Hall(12) normal
// (sum of twelve Philox lanes of counter (0, g, rep, 7<<24 | k/4)) * 2^-32 - 6.
__device__ double growth_rate(double r, double r_sd, uint32_t g, uint32_t rep, uint32_t key0, uint32_t key1) {
    if (r_sd == 0.0) return r;
    unsigned long long sum = 0;
#pragma unroll
    for (uint32_t k = 0; k < 3; ++k) {
        const uint4 d = philox(make_uint4(0u, g, rep, (kGrowth << 24) | k), key0, key1);
        sum += (unsigned long long)d.x + d.y + d.z + d.w;
    }
    const double u = __dmul_rn(__ull2double_rn(sum), 1.0 / 4294967296.0);
    const double z = __dsub_rn(u, 6.0);
    return __dadd_rn(r, __dmul_rn(r_sd, z));
}

__device__ uint32_t factor_q32(double R, double R_half) {
    const double den = __dadd_rn(R, R_half);
    const double q = __ddiv_rn(R, den);
    const double scaled = __dmul_rn(q, 4294967296.0);
    if (scaled >= 4294967294.0) return 0xFFFFFFFEu;
    if (!(scaled > 0.0)) return 0u;
    return __double2uint_rz(scaled);
}

}  // namespace
}  // namespace spg
