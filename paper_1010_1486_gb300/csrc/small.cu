// small.cu -- whole generation calls of a small lattice in one launch: one
// thread-block cluster runs every phase of every sweep (Sec. 2 update, Sec. 4
// schedule), with the hardware's cluster barrier between phases, and the
// measurements.
//
// A phase of a small lattice is latency: replayed from a graph, an 8^4 phase
// (2,048 links, one round of 64 warps) takes 3.6 us, of which the launch, the
// drain and the wait for the links are nearly all.  Here the links live in the
// shared memory of the cluster's CTAs for the whole launch (CTA c holds the
// even/odd indices [c L, (c + 1) L) of all eight arrays), so a phase is a
// barrier, reads of distributed shared memory and the chain from the staple to
// the store:
//   * what does not need the links -- the Philox blocks, the logarithms and
//     sines of the first two trials, the direction -- is computed a phase
//     ahead, where the links leave room for it by warps of their own (SPLIT:
//     as many again as have links), which the SM's schedulers run beside the
//     staples;
//   * the neighbours of a thread's links are tabulated once;
//   * the direction mu is a run-time value, so that all phases execute the
//     same instructions (one copy per mu keeps fetching them: the batch kernel
//     loses 6 to 12% to that).
// The chain is link for link that of the phase kernels, trial counts
// included, and the plaquette's binary32 partial sums are theirs.  With the
// links in global memory (through L2) instead, an 8^4 phase took 2.7 us.
// us per measured sweep, phase kernels replayed from a graph / here:
// Kennedy-Pendleton 4^4 38.0 / 15.8, 8^4 40.2 / 17.2, 8^3 x 16 40.1 / 24.0,
// 12^3 x 8 40.2 / 32.3; Creutz 8^4 63.0 / 32.5, 12^3 x 8 65.8 / 53.4.  Two links
// per thread lose (12^4: 40 / 54), so the limit is one: 8,192 links per phase.
#include <algorithm>
#include <cuda_runtime.h>

#include "kp_device.cuh"
#include "observables.cuh"
#include "staple.cuh"
#include "su2_device.cuh"
#include "su2_internal.h"

namespace su2 {

constexpr int kSmallThreads = 512;  // most threads per CTA
constexpr int kSmallCtas = 16;      // most CTAs of the cluster
constexpr int kSmallPerCta = 512;   // most links of a phase per CTA, a thread each
constexpr int kSmallLinks = kSmallCtas * kSmallPerCta;  // most links of a phase (V/2)
constexpr int kSmallSweeps = 256;   // sweeps per launch
constexpr int kRandomWords = 12;    // of a link's draw (Randoms)
// shared memory of a CTA per even/odd index: eight links, two parities' eight
// neighbours, two phases' randoms
constexpr size_t kSmallBytes = 8 * sizeof(float4) + 2 * 8 * sizeof(int) + 2 * kRandomWords * sizeof(uint32_t);

struct SmallParams {
    float4 *links;
    Geom g;
    RoundKeys rk;
    float beta, min_bk;
    uint32_t sweep;      // counter of the first sweep
    int first, nsweeps;  // sweeps first + 1 .. first + nsweeps of the call
    int measure_every, reunit_every;
    int overrelax;
    int max_trials;
    int log_per_cta;     // L = 2^log_per_cta links of a phase per CTA
    unsigned long long *trial_slots;
    unsigned int *flags;
    double *partials;    // [measured sweep of the launch][CTA][2]
    double *plaq, *poly;  // measurement slots of the first sweep of this launch
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// The cluster's links: element (array, eo) is at array L + (eo mod L) of CTA eo / L.
struct ClusterLinks {
    uint32_t base;  // this CTA's shared-memory address of the arrays
    int log_per_cta;
    __device__ __forceinline__ uint32_t address(int eo) const
    {
        uint32_t a;
        const uint32_t local = base + 16u * ((uint32_t)eo & ((1u << log_per_cta) - 1u));
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"((uint32_t)eo >> log_per_cta));
        return a;
    }
    __device__ __forceinline__ float4 load(uint32_t address, int array) const
    {
        float4 v;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "r"(address + ((uint32_t)array << (log_per_cta + 4)))
                     : "memory");
        return v;
    }
};

// The eighteen staple links of direction mu (run-time) from the neighbour
// table: nb[d L] and nb[(4 + d) L] hold the even/odd indices of x + d and x - d.
struct PhaseLinks {
    NuLinks n[3];
};

struct PhaseAddresses {
    uint32_t x, p, f[3], m[3], pm[3];  // x, x + mu, x + nu, x - nu, x + mu - nu
};

__device__ __forceinline__ PhaseAddresses phase_addresses(const ClusterLinks &cl, const int *nb, int eo, int mu)
{
    const int per = 1 << cl.log_per_cta, f_mu = nb[mu * per];
    PhaseAddresses a;
    a.x = cl.address(eo);
    a.p = cl.address(f_mu);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int nu = j + (j >= mu ? 1 : 0), b = nb[(4 + nu) * per];
        a.f[j] = cl.address(nb[nu * per]);
        a.m[j] = cl.address(b);
        a.pm[j] = cl.address(f_mu + b - eo);
    }
    return a;
}

__device__ __forceinline__ PhaseLinks load_phase_links(const ClusterLinks &cl, const PhaseAddresses &a, int mu, int parity)
{
    const int op = parity ^ 1;
    PhaseLinks l;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int nu = j + (j >= mu ? 1 : 0);
        l.n[j].nu_xp = cl.load(a.p, 2 * nu + op);
        l.n[j].mu_xn = cl.load(a.f[j], 2 * mu + op);
        l.n[j].nu_x = cl.load(a.x, 2 * nu + parity);
        l.n[j].nu_xpm = cl.load(a.pm[j], 2 * nu + parity);
        l.n[j].mu_xm = cl.load(a.m[j], 2 * mu + op);
        l.n[j].nu_xm = cl.load(a.m[j], 2 * nu + op);
    }
    return l;
}

// Their staple; sp: its terms of the directions below mu.
__device__ __forceinline__ float4 phase_staple(const PhaseLinks &l, int mu, float4 &sp)
{
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    sp = v;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        v = add_nu_terms(v, l.n[j]);
        if (j + 1 == mu) sp = v;
    }
    return v;
}

// A link outside the main path's range, by the checked operations: its trials
// (all of them) and direction.  Returns the trials used, negative if the cap
// was hit (the link keeps its value).
static __device__ __noinline__ int kp_out_of_range(const SmallParams &p, float4 v, uint32_t eo, uint32_t sweep,
                                                   uint32_t parity, uint32_t mu, float4 &out)
{
    const float k = __fsqrt_rn(qnorm2(v));
    const float bk = __fmul_rn(p.beta, k);
    if (!(bk >= kKpMinBk)) {
        const int n = heatbath_draw(v, p.beta, p.rk, eo, sweep, parity, mu, out);
        return n > 0 ? n : -kMaxTrials;
    }
    const float inv_k = __frcp_rn(k);
    const float4 ut = make_float4(__fmul_rn(v.x, inv_k), __fmul_rn(-v.y, inv_k), __fmul_rn(-v.z, inv_k),
                                  __fmul_rn(-v.w, inv_k));
    const float two_bk = __fmul_rn(2.0f, bk);
    float a0 = 0.0f;
    int t = 0;
    for (; t < p.max_trials; ++t)
        if (kp_trial(philox_rk(make_uint4(eo, sweep, stream_word(kKennedyPendleton, parity, mu), (uint32_t)t), p.rk),
                     two_bk, a0))
            break;
    if (t >= p.max_trials) return -p.max_trials;
    out = direction_update(
        a0, ut, philox_rk(make_uint4(direction_pair(eo), sweep, stream_word(kDirection, parity, mu), 0u), p.rk), eo);
    return t + 1;
}

// What a link's draw needs besides its staple.
struct Randoms {
    SpherePoint point;
    uint32_t w[8];  // Kennedy-Pendleton: numerators of trials 0 and 1 and their acceptance words; Creutz: blocks 0 and 1
};

template <int S>
__device__ __forceinline__ Randoms draw_randoms(const SmallParams &p, uint32_t eo, uint32_t sweep, uint32_t parity, int mu)
{
    Randoms r;
    uint4 wd = make_uint4(direction_pair(eo), sweep, stream_word(kDirection, parity, mu), 0u);
    if constexpr (S == SU2_SAMPLER_KP) {
        const uint32_t sw = stream_word(kKennedyPendleton, parity, mu);
        uint4 w0 = make_uint4(eo, sweep, sw, 0u), w1 = make_uint4(eo, sweep, sw, 1u);
        philox2_rk(w0, w1, p.rk);
        wd = philox_rk(wd, p.rk);
        r.w[0] = __float_as_uint(kp_numerator(w0));
        r.w[1] = __float_as_uint(kp_numerator(w1));
        r.w[2] = w0.w;
        r.w[3] = w1.w;
    } else {
        const uint32_t sw = stream_word(kCreutz, parity, mu);
        uint4 w0 = make_uint4(eo, sweep, sw, 0u), w1 = make_uint4(eo, sweep, sw, 1u);
        philox2_rk(w0, w1, p.rk);
        wd = philox_rk(wd, p.rk);
        r.w[0] = w0.x, r.w[1] = w0.y, r.w[2] = w0.z, r.w[3] = w0.w;
        r.w[4] = w1.x, r.w[5] = w1.y, r.w[6] = w1.z, r.w[7] = w1.w;
    }
    const bool odd = (eo & 1u) != 0u;
    r.point = sphere_point(uniform01(odd ? wd.z : wd.x), uniform01(odd ? wd.w : wd.y));
    return r;
}

// Handed from the warps that draw to the warps that have the links: word k of
// link i at buf[k L + i].
template <int S>
__device__ __forceinline__ void put_randoms(uint32_t *buf, int per, const Randoms &r)
{
    buf[0] = __float_as_uint(r.point.c);
    buf[per] = __float_as_uint(r.point.st);
    buf[2 * per] = __float_as_uint(r.point.sn);
    buf[3 * per] = __float_as_uint(r.point.cs);
#pragma unroll
    for (int k = 0; k < (S == SU2_SAMPLER_KP ? 4 : 8); ++k) buf[(4 + k) * per] = r.w[k];
}

template <int S>
__device__ __forceinline__ Randoms get_randoms(const uint32_t *buf, int per)
{
    Randoms r;
    r.point.c = __uint_as_float(buf[0]);
    r.point.st = __uint_as_float(buf[per]);
    r.point.sn = __uint_as_float(buf[2 * per]);
    r.point.cs = __uint_as_float(buf[3 * per]);
#pragma unroll
    for (int k = 0; k < (S == SU2_SAMPLER_KP ? 4 : 8); ++k) r.w[k] = buf[(4 + k) * per];
    return r;
}

// The heat bath of one link per lane.  Returns whether the link changes (to
// out); c: this lane's share of the plaquette sum as the phase kernel adds it.
template <int S>
__device__ __forceinline__ bool small_draw(const SmallParams &p, const Randoms &rnd, float4 v, float4 sp, bool valid,
                                           uint32_t eo, uint32_t sweep, uint32_t parity, int mu, float *s_warp,
                                           unsigned int &trials, float4 &out, float &c)
{
    if constexpr (S == SU2_SAMPLER_KP) {
        const float k = sqrt_in_range(qnorm2(v));
        const float bk = __fmul_rn(p.beta, k);
        const bool in_range = bk >= p.min_bk && bk <= kKpMaxBk;
        const float inv_k = rcp_in_range(k);
        const float4 ut = make_float4(__fmul_rn(v.x, inv_k), __fmul_rn(-v.y, inv_k), __fmul_rn(-v.z, inv_k),
                                      __fmul_rn(-v.w, inv_k));
        const float two_bk = __fmul_rn(2.0f, bk);
        float a0, a1;
        const bool ok0 = kp_candidate<true>(__uint_as_float(rnd.w[0]), rnd.w[2], two_bk, a0) && in_range;
        bool ok = kp_candidate<true>(__uint_as_float(rnd.w[1]), rnd.w[3], two_bk, a1) && in_range;
        int used = ok0 ? 1 : 2;
        a0 = ok0 ? a0 : a1;
        ok = ok || ok0;
        if (valid && in_range && !ok) {  // further trials
            const uint32_t sw = stream_word(kKennedyPendleton, parity, mu);
            while (!ok && used < p.max_trials)
                ok = kp_trial<true>(philox_rk(make_uint4(eo, sweep, sw, (uint32_t)used++), p.rk), two_bk, a0);
        }
        out = direction_from_point(a0, ut, rnd.point);
        if (valid && !in_range) {
            used = kp_out_of_range(p, v, eo, sweep, parity, (uint32_t)mu, out);
            ok = used > 0;
            used = ok ? used : -used;
        }
        if (valid) trials += (unsigned int)used;
        if (valid && !ok) atomicAdd(&p.flags[0], 1u);  // trial cap: the link keeps its old value
        // the phase kernel adds a link whose first trial was not accepted to
        // the sum of the lane that it waits for in the retry queue
        const float share = ok && valid ? qmul_re(out, sp) : 0.0f;
        c = ok0 ? share : 0.0f;
        const unsigned int parked = __ballot_sync(0xffffffffu, valid && !ok0);
        if (parked) {
            const int lane = threadIdx.x & 31;
            if (valid && !ok0) s_warp[__popc(parked & ((1u << lane) - 1u))] = share;
            __syncwarp();
            if (lane < __popc(parked)) c = __fadd_rn(c, s_warp[lane]);
            __syncwarp();
        }
        return valid && ok;
    } else {
        const uint32_t sw = stream_word(kCreutz, parity, mu);
        uint4 w = make_uint4(rnd.w[0], rnd.w[1], rnd.w[2], rnd.w[3]);
        const DrawSetup d = prepare_draw(v, p.beta);
        const int max_blocks = p.max_trials / 2;
        bool pending = valid, ok = false;
        float val = 0.0f;
        for (int blk = 0; __any_sync(0xffffffffu, pending); ++blk) {
            if (blk == 1) w = make_uint4(rnd.w[4], rnd.w[5], rnd.w[6], rnd.w[7]);
            if (blk > 1) w = philox_rk(make_uint4(eo, sweep, sw, (uint32_t)blk), p.rk);
            bool first;
            float x;
            const bool acc = creutz_pair(w, d.ibk, d.e, pending, first, x);
            if (pending && acc) {
                ok = true;
                val = x;
                trials += (unsigned int)(2 * blk + (first ? 1 : 2));
                pending = false;
            } else if (pending && blk + 1 >= max_blocks) {
                atomicAdd(&p.flags[0], 1u);  // trial cap: the link keeps its old value
                trials += (unsigned int)(2 * max_blocks);
                pending = false;
            }
        }
        out = direction_from_point(deferred_a0(val, d.ibk), d.ut, rnd.point);
        c = ok ? qmul_re(out, sp) : 0.0f;
        return ok;
    }
}

// A CTA has L threads with a link of every phase each, and for SPLIT as many
// again that draw the randoms of the next phase.
template <int S, bool SPLIT>
__global__ void __launch_bounds__(kSmallThreads, 1) small_sweep_kernel(const SmallParams p)
{
    extern __shared__ float4 s_links[];  // [2 mu + parity][L], then the neighbour table and the randoms
    __shared__ float s_warp[kSmallThreads / 32][32];
    __shared__ unsigned int s_trials[8];
    const int nthreads = blockDim.x, tid = threadIdx.x, lane = tid & 31;
    const int per = 1 << p.log_per_cta, eo0 = (int)blockIdx.x * per;
    const int vh = p.g.vh;
    int *const s_nb = (int *)(s_links + 8 * per);             // [parity][8][L]
    uint32_t *const s_random = (uint32_t *)(s_nb + 16 * per);  // [phase & 1][kRandomWords][L]
    const ClusterLinks cl{(uint32_t)__cvta_generic_to_shared(s_links), p.log_per_cta};
    const int links = max(0, min(per, vh - eo0));  // of this CTA
    const int phases = 8 * (1 + p.overrelax);
    if (tid < 8) s_trials[tid] = 0u;
    for (int i = tid; i < per; i += nthreads) {
        const int eo = min(eo0 + i, vh - 1);
        for (int a = 0; a < 8; ++a) s_links[a * per + i] = p.links[(size_t)a * vh + eo];
        for (int parity = 0; parity < 2; ++parity) {
            const Coord x = eo_to_coord(p.g, eo, parity);
            int *const nb = s_nb + parity * 8 * per + i;
            nb[0] = eo_fwd<0>(p.g, x, eo);
            nb[per] = eo_fwd<1>(p.g, x, eo);
            nb[2 * per] = eo_fwd<2>(p.g, x, eo);
            nb[3 * per] = eo_fwd<3>(p.g, x, eo);
            nb[4 * per] = eo + eo_bwd_offset<0>(p.g, x);
            nb[5 * per] = eo + eo_bwd_offset<1>(p.g, x);
            nb[6 * per] = eo + eo_bwd_offset<2>(p.g, x);
            nb[7 * per] = eo + eo_bwd_offset<3>(p.g, x);
        }
    }
    __syncthreads();  // the table
    const bool draws = SPLIT && tid >= per;  // warp-uniform: L is a multiple of 32
    const int i = tid & (per - 1);
    const bool valid = !draws && i < links;
    const int eo = min(eo0 + i, vh - 1);
    // the randoms of phase ph (a heat bath's) of the launch's sweep s, into their buffer
    auto draw_ahead = [&](int s, int ph) {
        put_randoms<S>(s_random + (ph & 1) * kRandomWords * per + i, per,
                       draw_randoms<S>(p, (uint32_t)eo, p.sweep + (uint32_t)s, (uint32_t)(ph & 1), ph >> 1));
    };
    if (draws) draw_ahead(0, 0);
    cluster_arrive();  // every wait below is for the latest arrival
    int slot = 0;
#pragma unroll 1
    for (int s = 0; s < p.nsweeps; ++s) {
        const int number = p.first + s + 1;
        const bool measure = p.measure_every > 0 && number % p.measure_every == 0;
        const bool reunit = p.reunit_every > 0 && number % p.reunit_every == 0;
        const uint32_t sweep = p.sweep + (uint32_t)s;
        double plaq = 0.0, poly = 0.0;
#pragma unroll 1
        for (int ph = 0; ph < phases; ++ph) {
            const int mu = (ph >> 1) & 3, parity = ph & 1;
            if (draws) {
                cluster_wait();
                if (ph + 1 < 8) draw_ahead(s, ph + 1);
                if (ph + 1 == phases && s + 1 < p.nsweeps) draw_ahead(s + 1, 0);
            } else {
                const bool meas = measure && !reunit && ph >= 8 * p.overrelax && parity == 1 && mu > 0;
                const PhaseAddresses at = phase_addresses(cl, s_nb + parity * 8 * per + i, eo, mu);
                Randoms rnd;
                if (!SPLIT && ph < 8) rnd = draw_randoms<S>(p, (uint32_t)eo, sweep, (uint32_t)parity, mu);
                cluster_wait();
                const PhaseLinks l = load_phase_links(cl, at, mu, parity);
                if (SPLIT && ph < 8) rnd = get_randoms<S>(s_random + parity * kRandomWords * per + i, per);
                float4 *const own = s_links + (2 * mu + parity) * per + i;
                float4 sp, out;
                const float4 v = phase_staple(l, mu, sp);
                float c;
                if (ph < 8) {
                    unsigned int trials = 0;
                    if (small_draw<S>(p, rnd, v, sp, valid, (uint32_t)eo, sweep, (uint32_t)parity, mu, s_warp[tid >> 5],
                                      trials, out, c))
                        *own = out;
                    const unsigned int wsum = __reduce_add_sync(0xffffffffu, trials);
                    if (lane == 0) atomicAdd(&s_trials[ph], wsum);
                } else {
                    const float4 ut = staple_direction(v);
                    out = qmul(qmul(ut, qdag(*own)), ut);
                    if (valid) *own = out;
                    c = valid ? qmul_re(out, sp) : 0.0f;
                }
                if (meas) plaq += (double)c;
            }
            cluster_arrive();
        }
        if (!measure && !reunit) continue;  // uniform over the cluster
        cluster_wait();
        if (reunit) {
            for (int q = tid; q < 8 * per; q += nthreads) {
                const float4 a = s_links[q];
                const float r = __fsqrt_rn(qnorm2(a));
                s_links[q] = make_float4(__fdiv_rn(a.x, r), __fdiv_rn(a.y, r), __fdiv_rn(a.z, r), __fdiv_rn(a.w, r));
            }
            cluster_arrive();
            if (!measure) continue;
            cluster_wait();
            // the plaquettes of this CTA's sites, as site_plaquette
            for (int q = tid; q < 2 * per; q += nthreads) {
                const int parity = q >> p.log_per_cta, k = q & (per - 1), op = parity ^ 1;
                if (k >= links) continue;
                uint32_t a[4];
#pragma unroll
                for (int mu = 0; mu < 4; ++mu) a[mu] = cl.address(s_nb[(parity * 8 + mu) * per + k]);
                float sum = 0.0f;
#pragma unroll
                for (int mu = 0; mu < 4; ++mu)
#pragma unroll
                    for (int nu = mu + 1; nu < 4; ++nu) {
                        const float4 t = qmul(qmul(s_links[(2 * mu + parity) * per + k], cl.load(a[mu], 2 * nu + op)),
                                              qdag(cl.load(a[nu], 2 * mu + op)));
                        sum = __fadd_rn(sum, qmul_re(t, qdag(s_links[(2 * nu + parity) * per + k])));
                    }
                plaq += (double)sum;
            }
        }
        // Polyakov loop: four lanes per spatial site, a quarter of the time
        // extent each, combined as (P0 P1)(P2 P3)
        const int len = (p.g.nt + 3) / 4;
        for (int q = (int)blockIdx.x * nthreads + tid; q < ((4 * p.g.vs + 31) & ~31); q += (int)gridDim.x * nthreads) {
            const int xs = min(q >> 2, p.g.vs - 1), t0 = min((q & 3) * len, p.g.nt), t1 = min(t0 + len, p.g.nt);
            const uint32_t r1 = fastdiv((uint32_t)xs, p.g.div_ns), z = fastdiv(r1, p.g.div_ns);
            const int p0 = (int)(((uint32_t)xs - r1 * (uint32_t)p.g.ns) + (r1 - z * (uint32_t)p.g.ns) + z) & 1;
            float4 u = make_float4(1.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 4
            for (int t = t0; t < t1; ++t)
                u = qmul(u, cl.load(cl.address((t * p.g.vs + xs) >> 1), 6 + ((p0 + t) & 1)));
            float4 o;
#pragma unroll
            for (int step = 1; step <= 2; ++step) {
                o.x = __shfl_down_sync(0xffffffffu, u.x, step);
                o.y = __shfl_down_sync(0xffffffffu, u.y, step);
                o.z = __shfl_down_sync(0xffffffffu, u.z, step);
                o.w = __shfl_down_sync(0xffffffffu, u.w, step);
                u = qmul(u, o);
            }
            if ((q & 3) == 0 && (q >> 2) < p.g.vs) poly += (double)u.x;
        }
        cluster_arrive();  // the links may change again; the sums are this CTA's own
        plaq = block_sum(plaq);
        poly = block_sum(poly);
        if (tid == 0) {
            p.partials[2 * (slot * gridDim.x + blockIdx.x)] = plaq;
            p.partials[2 * (slot * gridDim.x + blockIdx.x) + 1] = poly;
        }
        ++slot;
    }
    cluster_wait();  // nobody reads this CTA's links any more
    for (int q = tid; q < links; q += nthreads)
        for (int a = 0; a < 8; ++a) p.links[(size_t)a * vh + eo0 + q] = s_links[a * per + q];
    __syncthreads();
    if (tid < 8 && s_trials[tid])
        atomicAdd(&p.trial_slots[tid * kTrialSlots + (blockIdx.x & (kTrialSlots - 1))], (unsigned long long)s_trials[tid]);
    // the measurements: the CTAs' sums in order
    cluster_arrive();
    cluster_wait();
    if (blockIdx.x == 0)
        for (int m = tid; m < slot; m += nthreads) {
            double plaq = 0.0, poly = 0.0;
            for (unsigned int b = 0; b < gridDim.x; ++b) {
                plaq += __ldcg(p.partials + 2 * (m * gridDim.x + b));
                poly += __ldcg(p.partials + 2 * (m * gridDim.x + b) + 1);
            }
            p.plaq[m] = plaq * (1.0 / (12.0 * (double)vh));
            p.poly[m] = poly * (1.0 / (double)p.g.vs);
        }
}

bool small_lattice(const su2_lattice *lat)
{
    return !lat->timing && lat->vh <= kSmallLinks;
}

su2_status small_sweeps(su2_lattice *lat, int nsweeps, int measure_every, int reunit_every, double *plaq, double *poly,
                        bool *done)
{
    *done = false;
    SmallParams p;
    p.links = lat->links;
    p.g = geom_of(lat);
    p.rk = make_round_keys(lat->seed);
    p.beta = (float)lat->beta;
    p.min_bk = kp_min_bk(p.beta);
    p.measure_every = measure_every;
    p.reunit_every = reunit_every;
    p.overrelax = lat->overrelax;
    p.max_trials = lat->max_trials;
    p.trial_slots = lat->scratch.trials;
    p.flags = lat->scratch.flags;
    p.partials = lat->scratch.partials;
    // as many SMs as the links fill with four warps each, up to the cluster's
    // sixteen, then more warps per SM
    int per = 128;
    p.log_per_cta = 7;
    while (per < kSmallPerCta && per * kSmallCtas < lat->vh) per *= 2, ++p.log_per_cta;
    const int ctas = (lat->vh + per - 1) / per;
    const bool split = 2 * per <= kSmallThreads;
    const int threads = split ? 2 * per : per;
    const size_t smem = kSmallBytes * (size_t)per;
    const bool kp = lat->sampler == SU2_SAMPLER_KP;
    const auto kernel = kp ? (split ? small_sweep_kernel<SU2_SAMPLER_KP, true> : small_sweep_kernel<SU2_SAMPLER_KP, false>)
                           : (split ? small_sweep_kernel<SU2_SAMPLER_CREUTZ, true>
                                    : small_sweep_kernel<SU2_SAMPLER_CREUTZ, false>);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = lat->stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = ctas;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int &room = lat->small_room[lat->sampler];  // 0 not asked yet, 1 the cluster fits this device, 2 it does not
    if (room == 0) {
        SU2_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(kSmallBytes * kSmallPerCta)));
        SU2_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            clusters = 0;
        }
        room = clusters > 0 ? 1 : 2;
    }
    if (room == 2) return SU2_OK;
    for (int first = 0; first < nsweeps; first += kSmallSweeps) {
        p.first = first;
        p.nsweeps = std::min(kSmallSweeps, nsweeps - first);
        p.sweep = lat->sweep;
        const int m = measure_every > 0 ? first / measure_every : 0;
        p.plaq = plaq ? plaq + m : nullptr;
        p.poly = poly ? poly + m : nullptr;
        SU2_CUDA(cudaLaunchKernelEx(&cfg, kernel, p));
        lat->sweep += (uint32_t)p.nsweeps;
    }
    *done = true;
    return SU2_OK;
}

}  // namespace su2
