// observables.cu -- mean plaquette and Polyakov loop with their global sums
// (Sec. 4 of Cardoso & Bicudo: per-site plaquette and Polyakov kernels and a
// kernel summing over all sites, here fused into one kernel each).
//
// Per-site values are binary32 (same operation order as the updates); the
// sum is binary64: warp shuffles, then one partial per block, then the last
// block to finish adds the partials in block order, so the result does not
// depend on the order in which blocks run.
#include <algorithm>

#include "observables.cuh"
#include "plaquette_plan.h"
#include "su2_device.cuh"
#include "su2_internal.h"

namespace su2 {

// Mean plaquette.  A thread takes one spatial site and walks along t: the
// links U_0..U_2 that it reads at t + 1 for the planes with t are its own links
// of the next step, and the block's 384 consecutive pairs of sites (both
// spatial parities, a warp for 32 pairs of one parity: every load is 512
// contiguous bytes) find most of their neighbours in y in L1, where the block
// itself read them.  Thirteen loads per site remain, all in flight at once.
// One site per thread in lexicographic order (sixteen loads, two runs of 256
// bytes each) was bound by L1 wavefronts (88%), and the same by even/odd order
// by the traffic from L2 (87 us, 12.7 TB/s).  48^4: 100 -> 90 us per call, 82 us
// (ncu) in the kernel, which waits for its loads (24 warps per SM, 80
// registers); splitting the planes into two groups of loads, one in flight
// while the other is computed, spills (102 us) or halves the warps (106 us).
constexpr int kPlaqThreads = 2 * kPlaqPairs;    // one block per SM

// dst (+ *idx when idx is given: the measurement slot of a graph replay)
__global__ void __launch_bounds__(kPlaqThreads, 1) plaquette_kernel(const float4 *__restrict__ L, Geom g, PlaquettePlan pl,
                                                                  double *__restrict__ partials,
                                                                  unsigned int *__restrict__ ticket,
                                                                  double *__restrict__ dst,
                                                                  const uint32_t *__restrict__ idx)
{
    double acc = 0.0;
    const int half = g.vs >> 1;
    const int sp = (int)threadIdx.x >= kPlaqPairs;  // spatial parity, warp-uniform
#pragma unroll 1
    for (int item = (int)blockIdx.x; item < pl.items; item += (int)gridDim.x) {
        const int chunk = item / pl.pair_blocks;
        const int j = (item - chunk * pl.pair_blocks) * kPlaqPairs + (int)threadIdx.x - sp * kPlaqPairs;
        const int t0 = chunk * pl.t_chunk, t1 = min(t0 + pl.t_chunk, g.nt);
        if (j >= half) continue;
        const uint32_t r1 = fastdiv(2u * (uint32_t)j, g.div_ns), z = fastdiv(r1, g.div_ns);
        const int y = (int)(r1 - z * (uint32_t)g.ns);
        const int x = 2 * j - (int)r1 * g.ns + ((y + (int)z + sp) & 1);
        // the pair indices of x + 0, x + 1, x + 2 (at the other parity)
        const int f[3] = {j + (x & 1) - (x == g.ns - 1 ? g.ns >> 1 : 0),
                          y == g.ns - 1 ? j - (g.wrap[1] >> 1) : j + (g.stride[1] >> 1),
                          (int)z == g.ns - 1 ? j - (g.wrap[2] >> 1) : j + (g.stride[2] >> 1)};
        float4 u[4];
#pragma unroll
        for (int mu = 0; mu < 3; ++mu) u[mu] = __ldg(L + link_index(g, mu, (sp + t0) & 1, t0 * half + j));
#pragma unroll 1
        for (int t = t0; t < t1; ++t) {
            const int parity = (sp + t) & 1, op = parity ^ 1, at = t * half;
            const int ahead = (t == g.nt - 1 ? 0 : at + half) + j;
            float4 b[3][4], c[3];  // b[mu][nu] = U_nu(x + mu); U_mu(x + nu) for nu < 3 is b[nu][mu]; c[mu] = U_mu(x + t)
            u[3] = __ldg(L + link_index(g, 3, parity, at + j));
#pragma unroll
            for (int mu = 0; mu < 3; ++mu) {
                c[mu] = __ldg(L + link_index(g, mu, op, ahead));
#pragma unroll
                for (int nu = 0; nu < 4; ++nu)
                    if (nu != mu) b[mu][nu] = __ldg(L + link_index(g, nu, op, at + f[mu]));
            }
            float sum = 0.0f;
#pragma unroll
            for (int mu = 0; mu < 3; ++mu)
#pragma unroll
                for (int nu = mu + 1; nu < 4; ++nu)
                    sum = __fadd_rn(sum, qmul_re(qmul(qmul(u[mu], b[mu][nu]), qdag(nu == 3 ? c[mu] : b[nu][mu])),
                                                 qdag(u[nu])));
            acc += (double)sum;
#pragma unroll
            for (int mu = 0; mu < 3; ++mu) u[mu] = c[mu];
        }
    }
    const double total = block_sum(acc);
    finish_reduction(total, partials, ticket, idx ? dst + *idx : dst, 1.0 / (12.0 * (double)g.vh));
}

// (1/2) Tr of U_3(x,0) U_3(x,1) ... U_3(x,Nt-1).  A block of kPolySeg warps
// takes 32 consecutive spatial sites at a time; warp s multiplies, left to
// right, the links of the s-th quarter of the time extent for each of the 32
// sites (each load instruction reads one time slice: 32 consecutive sites,
// two runs of 256 B), with all of a quarter's loads (up to kPolyBatch) in
// flight at once.  Warp 0 then combines the quarters through shared memory
// as (P0 P1)(P2 P3).  Short quarters are padded with the identity, which
// multiplies exactly.
constexpr int kPolySeg = 4;                  // warps per block: quarters of the time extent
constexpr int kPolyThreads = 32 * kPolySeg;  // block size
constexpr int kPolyBatch = 12;               // loads in flight per lane (Nt = 48: one batch)

// PLAQ: the kernel of a measuring sweep also sums the fused-plaquette slots
// (fused.n[r] of region r): each block a share of every region, and the last
// block the block sums in block order, into plaq_dst (scaled by plaq_scale),
// beside the Polyakov loop; it then advances the counters of a graph replay
// (ctr).  `partials` holds 2 gridDim.x doubles and must not
// overlap the slots.
struct FusedSlots {
    const double *slots;
    int n[6];
};

template <bool PLAQ>
__global__ void __launch_bounds__(kPolyThreads) polyakov_kernel(const float4 *__restrict__ L, Geom g,
                                                               double *__restrict__ partials,
                                                               unsigned int *__restrict__ ticket,
                                                               double *__restrict__ dst,
                                                               const uint32_t *__restrict__ idx,
                                                               const FusedSlots fused,
                                                               double *__restrict__ plaq_dst, double plaq_scale,
                                                               uint32_t *__restrict__ ctr)
{
    __shared__ float4 s_part[kPolySeg][32];
    float acc = 0.0f;  // per-thread partial in binary32; the block and grid sums are binary64
    const int lane = threadIdx.x & 31;
    const int seg = threadIdx.x >> 5;
    const int len = (g.nt + kPolySeg - 1) / kPolySeg;
    const int t_begin = min(seg * len, g.nt);
    const int t_end = min(t_begin + len, g.nt);
    const float4 one = make_float4(1.0f, 0.0f, 0.0f, 0.0f);
    // the slots first: their loads are in flight beside those of the links (and
    // the two sums of a block and of the grid side by side: 604.6 -> 601.0 us
    // per measured 48^4 sweep, 53.9 -> 53.3 on 32^3 x 4)
    double fused_sum = 0.0;
    if (PLAQ) {
#pragma unroll
        for (int r = 0; r < 6; ++r)
            for (int i = (int)blockIdx.x * kPolyThreads + (int)threadIdx.x; i < fused.n[r];
                 i += (int)gridDim.x * kPolyThreads)
                fused_sum += fused.slots[r * kFusedSlots + i];
    }
    // block-uniform loop over groups of 32 sites
    for (int base = blockIdx.x * 32; base < g.vs; base += gridDim.x * 32) {
        const int xs = min(base + lane, g.vs - 1);
        const int rest = xs / g.ns;
        const int x = xs - rest * g.ns;
        const int y = rest % g.ns;
        const int z = rest / g.ns;
        const int p0 = (x + y + z) & 1;
        // a quarter of up to kPolyBatch links (Nt <= 4 kPolyBatch) is one
        // batch of unconditional loads (the index clamped to the quarter),
        // all issued before the first product; longer quarters loop
        auto batch = [&](float4 p, int t) {
            float4 q[kPolyBatch];
#pragma unroll
            for (int j = 0; j < kPolyBatch; ++j) {
                const int tj = min(t + j, t_end - 1);
                const int64_t lex = (int64_t)tj * g.vs + xs;
                q[j] = __ldg(L + link_index(g, 3, (p0 + tj) & 1, (int)(lex >> 1)));
            }
#pragma unroll
            for (int j = 0; j < kPolyBatch; ++j) p = qmul(p, t + j < t_end ? q[j] : one);
            return p;
        };
        float4 p = t_begin < t_end ? batch(one, t_begin) : one;
        for (int t = t_begin + kPolyBatch; t < t_end; t += kPolyBatch) p = batch(p, t);
        s_part[seg][lane] = p;
        __syncthreads();
        if (seg == 0) {
            const float4 p01 = qmul(s_part[0][lane], s_part[1][lane]);
            const float4 p23 = qmul(s_part[2][lane], s_part[3][lane]);
            if (base + lane < g.vs) acc = __fadd_rn(acc, qmul(p01, p23).x);
        }
        __syncthreads();
    }
    if (!PLAQ) {
        finish_reduction(block_sum((double)acc), partials, ticket, idx ? dst + *idx : dst, 1.0 / (double)g.vs);
        return;
    }
    double total_sum = (double)acc;
    block_sum2(total_sum, fused_sum);
    __shared__ bool last;
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = total_sum;
        partials[gridDim.x + blockIdx.x] = fused_sum;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double vp = 0.0, vq = 0.0;
    for (unsigned int b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
        vp += ((volatile double *)partials)[b];
        vq += ((volatile double *)partials)[gridDim.x + b];
    }
    block_sum2(vp, vq);
    if (threadIdx.x == 0) {
        const uint32_t slot = ctr ? ctr[1] : 0u;
        dst[slot] = vp * (1.0 / (double)g.vs);
        plaq_dst[slot] = vq * plaq_scale;
        *ticket = 0u;
        if (ctr) {
            ctr[0] += 1u;
            ctr[1] = slot + 1u;
        }
    }
}

su2_status launch_plaquette(su2_lattice *lat, double *dst)
{
    const Geom g = geom_of(lat);
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, lat->device);
    const PlaquettePlan pl = plaquette_plan(g.vs, lat->nt, sms);
    plaquette_kernel<<<pl.grid, kPlaqThreads, 0, lat->stream>>>(lat->links, g, pl, lat->scratch.partials,
                                                                lat->scratch.ticket, dst,
                                                                lat->capturing ? lat->d_ctr + 1 : nullptr);
    SU2_CUDA(cudaGetLastError());
    return SU2_OK;
}

su2_status fused_begin(su2_lattice *lat)
{
    if (lat->scratch.partials_cap < kFusedRegion) {
        set_last_error("reduction scratch too small for the fused plaquette");
        return SU2_E_INVAL;
    }
    lat->fused_part = lat->scratch.partials;
    for (int &n : lat->fused_blocks) n = 0;
    return SU2_OK;
}

su2_status launch_polyakov(su2_lattice *lat, double *dst)
{
    const Geom g = geom_of(lat);
    const int grid = grid_for(g.vs, 32, std::min(lat->scratch.partials_cap, 152 * 8));
    polyakov_kernel<false><<<grid, kPolyThreads, 0, lat->stream>>>(lat->links, g, lat->scratch.partials,
                                                                     lat->scratch.ticket + 1, dst,
                                                                     lat->capturing ? lat->d_ctr + 1 : nullptr,
                                                                     FusedSlots(), nullptr, 0.0, nullptr);
    SU2_CUDA(cudaGetLastError());
    return SU2_OK;
}

su2_status fused_finish_with_polyakov(su2_lattice *lat, double *plaq_dst, double *poly_dst)
{
    const Geom g = geom_of(lat);
    const int grid = grid_for(g.vs, 32, 152 * 8);
    if (lat->scratch.partials_cap < kFusedRegion + 2 * grid) {
        set_last_error("reduction scratch too small for the fused plaquette");
        return SU2_E_INVAL;
    }
    lat->fused_part = nullptr;
    FusedSlots fused;
    fused.slots = lat->scratch.partials;
    std::copy(lat->fused_blocks, lat->fused_blocks + 6, fused.n);
    polyakov_kernel<true><<<grid, kPolyThreads, 0, lat->stream>>>(
        lat->links, g, lat->scratch.partials + kFusedRegion, lat->scratch.ticket + 1, poly_dst, nullptr, fused, plaq_dst,
        1.0 / (6.0 * (double)lat->vol), lat->capturing ? lat->d_ctr : nullptr);
    SU2_CUDA(cudaGetLastError());
    return SU2_OK;
}

}  // namespace su2

using namespace su2;

// Runs an observable and brings its value to the host: the kernel writes it
// into a page-locked page itself, or, when none is free, to *dev to be copied.
static su2_status read_value(su2_lattice *lat, su2_status (*launch)(su2_lattice *, double *), double *dev, double *out)
{
    HostPage page(lat->stream);
    su2_status st = launch(lat, page.p ? (double *)page.p : dev);
    if (st != SU2_OK) return st;
    if (!page.p) SU2_CUDA(cudaMemcpyAsync(out, dev, sizeof(double), cudaMemcpyDeviceToHost, lat->stream));
    SU2_CUDA(cudaStreamSynchronize(lat->stream));
    page.settled();
    if (page.p) *out = *(const double *)page.p;
    return SU2_OK;
}

extern "C" {

su2_status su2_plaquette(su2_lattice *lat, double *out)
{
    if (!lat || !out) return SU2_E_INVAL;
    DeviceGuard guard(lat->device);
    return read_value(lat, launch_plaquette, lat->scratch.result, out);
}

su2_status su2_polyakov(su2_lattice *lat, double *out)
{
    if (!lat || !out) return SU2_E_INVAL;
    DeviceGuard guard(lat->device);
    return read_value(lat, launch_polyakov, lat->scratch.result + 1, out);
}

}  // extern "C"
