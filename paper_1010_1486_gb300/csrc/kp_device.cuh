// kp_device.cuh -- the Kennedy-Pendleton a0 trial (Phys. Lett. B 156 (1985)
// 393), shared by the single-lattice and the batched phase kernels.
//
// With a0 = 1 - 2u the heat-bath law of Sec. 2 becomes u^{1/2} sqrt(1 - u)
// exp(-2 beta k u) on [0, 1]; a trial draws u = -(ln r1 + cos^2(2 pi r2) ln r3)
// / (2 beta k) and accepts iff u <= 1 and r4^2 <= 1 - u.  Trial t uses block t
// of the Kennedy-Pendleton stream; links with beta k < 2 are drawn by
// Creutz's method instead.
#pragma once

#include "su2_device.cuh"

namespace su2 {

constexpr float kKpMinBk = 2.0f;
// A link whose beta k lies in [lo, hi] is drawn with the range-limited
// operations: hi = 2^60, and lo = 2 or, for beta above 2^31, beta 2^-30, so
// that k (of the staple norm's square root) is within sqrt_in_range too.
// Others take the checked operations, in the retry queue.
constexpr float kKpMaxBk = 0x1p60f;
__host__ __device__ inline float kp_min_bk(float beta)
{
    const float lo = beta * 0x1p-30f;
    return lo > kKpMinBk ? lo : kKpMinBk;
}
constexpr uint32_t kKennedyPendleton = 5u;  // stream kind of the trials

// The part of a trial that does not need the staple: cos^2(2 pi r2) ln r3 + ln r1.
template <bool CHECKED_LOG = false>
__device__ __forceinline__ float kp_numerator(uint4 w)
{
    float sn, cs;
    sincos_2pi(uniform01(w.y), sn, cs);
    return __fmaf_rn(__fmul_rn(cs, cs), log_series<CHECKED_LOG>(uniform_log(w.z)),
                     log_series<CHECKED_LOG>(uniform_log(w.x)));
}

// ... and the rest: a0 = 1 - 2 u, and whether it is accepted.
template <bool IN_RANGE>
__device__ __forceinline__ bool kp_candidate(float num, uint32_t w3, float two_bk, float &a0)
{
    const float lam2 = IN_RANGE ? div_in_range(-num, two_bk) : __fdiv_rn(-num, two_bk);
    const float r4 = uniform01(w3);
    a0 = __fmaf_rn(-2.0f, lam2, 1.0f);
    return lam2 <= 1.0f && __fmul_rn(r4, r4) <= __fsub_rn(1.0f, lam2);
}

// One trial (block t of the KP stream).  IN_RANGE: 2 beta k is at most 2^61.
// The numerator is 0 or above 2^-67 (|ln| >= 2^-24 unless zero, cos^2 >= 2^-43),
// so from beta k = 2^22 on the quotient can fall below the range in which
// div_in_range is correctly rounded.  Both forms are then below 2^-89, and the
// trial takes only 1 - 2 l and 1 - l of it, which are 1.
template <bool IN_RANGE = false, bool CHECKED_LOG = false>
__device__ __forceinline__ bool kp_trial(uint4 w, float two_bk, float &a0)
{
    return kp_candidate<IN_RANGE>(kp_numerator<CHECKED_LOG>(w), w.w, two_bk, a0);
}

}  // namespace su2
