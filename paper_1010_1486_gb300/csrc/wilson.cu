// wilson.cu -- space-time Wilson loops W(R, T) (the observables that come
// after the Sec. 4 plaquette and Polyakov loop; not in the paper).
//
// For a site x, a spatial direction i and extents R (along i), T (along t):
//   S_R(y) = U_i(y) U_i(y+i) ... U_i(y+(R-1)i),  T_T(y) = U_t(y) ... U_t(y+(T-1)t),
//   A = S_R(x) T_T(x+Ri),  B = T_T(x) S_R(x+Tt),  loop = (1/2) Tr A B^dag = A . B,
// line products left to right, binary32 per loop (the link-arithmetic
// contract); the mean over x and i = 0, 1, 2 is exact to 2^-44 per loop in
// fixed point (wilson_tile_kernel), or binary64 (wilson_kernel) for few small
// loops, and for configurations whose loops leave the fixed-point range.
#include <algorithm>

#include "observables.cuh"
#include "su2_device.cuh"
#include "su2_internal.h"

namespace su2 {

constexpr int kWilsonThreads = 256;
constexpr int kWilsonMaxR = 16;
constexpr int kWilsonMaxT = 64;

// ------------------------------------------------------- tiled kernel
// All loops of an (i, t) plane stay inside the plane, so a block takes a tile
// of bx x bt sites of one plane (one site per thread) and a chunk of up to
// 8 x 8 extents (R, T) and works from shared memory:
//   * the lines S_R of the rows the tile's tops reach, for every R of the
//     chunk, are formed once (s_buf);
//   * T_T is extended by one link per step of T and published with the
//     columns x + R next to the tile (tt_buf, double buffered: one block
//     barrier per step);
//   * a loop is then two shared-memory loads, the products A and B and their
//     scalar product: 36 of its about 50 instructions.
// The walk it replaces formed T_T(x + Ri) again for every R and T from global
// loads (T + 2 loads and T + 2 products per loop), and added every loop in
// binary64, of which this chip starts two per clock and SM.  Here the loop
// value x is split exactly into integers, x = h 2^-21 + l 2^-43 (l rounded to
// nearest), by adding and subtracting 6 = 1.5 2^2, whose binary32 neighbours
// lie 2^-21 apart; the warp adds h and l with integer reductions, the block
// and the grid with integer atomics, so the sum does not depend on any order
// and is within 2^-44 per loop of the exact one.  (A loop of 2^-20 or more is a
// multiple of 2^-43 and taken exactly; of the smaller ones, one in a million, the
// mean keeps its error below that of a binary64 sum, about 2^-53 per addition.)
// |x| < 2 is required (unit links give |x| <= 1); a loop outside (links that are not unit, NaN) sets
// *flag, and the host then takes the binary64 path.
// Bound: instruction issue (71% of the slots; 82 warp instructions per 32
// loops, the tile's preparation included).  24^4, all loops up to 8 x 8: 1243
// -> 217 us per call, of it 189 us (ncu) in this kernel.  Fewer instructions
// alone do not help: loops in pairs (R, R + 1) with packed multiply-adds took
// 205 to 246 us at 24^4 and 3% more at 48^4.
constexpr int kLoopChunk = 8;          // extents R and T per block
constexpr int kTileThreads = 256;      // most sites of a tile
constexpr int kTileMaxBx = 64;         // most columns of a tile
constexpr float kSplit = 6.0f;         // its neighbours lie 2^-21 apart
constexpr unsigned int kSplitBits = 0x40C00000u;

struct LoopTiles {
    int bx, bt;          // tile extents along i and t
    int rc, tc;          // most extents R and T of a chunk of this call
    int nx, nt, nr, ntc;  // tiles along i, along t, chunks of R, chunks of T
};

__device__ __forceinline__ int wrap_once(int c, int extent) { return c >= extent ? c - extent : c; }

// Shared memory of a tile with extents bx x bt for chunks of up to rc x tc
// extents, in float4: [0] the two T_T buffers, which first hold the staged U_i
// (rows t0 + tc0 .. + bt + tc - 1, columns x0 .. x0 + ucols - 1, all of them when
// they cover the extent), [1] the staged U_t (one row less), [2] s_buf.  (Laid
// out for 8 x 8 extents whatever the call asked for, a tile of 56 columns left
// room for one block per SM: 56^4, R = T = 1, 3.3 ms instead of 1.3.)
struct TileSmem {
    int ucols, ut, s, total;
};

// float4 per site of s_buf: an odd pitch keeps 16-byte reads conflict-free
__host__ __device__ constexpr int top_pitch(int rc) { return rc | 1; }

__host__ __device__ constexpr TileSmem tile_smem(int bx, int bt, int rc, int tc, int ns, int r0)
{
    TileSmem m = {};
    m.ucols = bx + r0 + rc < ns ? bx + r0 + rc : ns;
    const int buf = 2 * bt * (bx + rc), ui = (bt + tc) * m.ucols;
    m.ut = buf > ui ? buf : ui;
    m.s = m.ut + (bt + tc - 1) * m.ucols;
    m.total = m.s + top_pitch(rc) * (bt + tc) * bx;
    return m;
}

// The most that a tile takes: kTileMaxBx columns of a longer row, the second
// chunk of R.  (Narrower tiles have more rows, but at most 256 sites all the
// same, and their staged rows end at the extent.)
constexpr size_t kTileMaxSmem =
    sizeof(float4) * (size_t)tile_smem(kTileMaxBx, kTileThreads / kTileMaxBx, kLoopChunk, kLoopChunk, 1 << 20,
                                       kWilsonMaxR - kLoopChunk)
                         .total;

// FULL: the chunk has all eight R (no test per R in the inner loop).
template <bool FULL>
__global__ void __launch_bounds__(kTileThreads, 3)
    wilson_tile_kernel(const float4 *__restrict__ L, Geom g, LoopTiles tl, int rmax, int tmax,
                       unsigned long long *__restrict__ slots, int nslots, unsigned int *__restrict__ flag)
{
    extern __shared__ float4 sm[];
    // [T][R][h, l] of the chunk, modulo 2^32; starts at minus what the bits of
    // 6 add up to over the block's warps
    __shared__ unsigned int s_sum[2 * kLoopChunk * kLoopChunk];
    const int rc = FULL ? kLoopChunk : tl.rc, tp = top_pitch(rc);
    const int pitch = tl.bx + rc;  // a T_T row: the tile's columns, then x + R
    const int buf_len = tl.bt * pitch;
    uint32_t b = blockIdx.x;
    const int r0 = (int)(b % (uint32_t)tl.nr) * kLoopChunk;
    b /= (uint32_t)tl.nr;
    const int tc0 = (int)(b % (uint32_t)tl.ntc) * kLoopChunk;
    b /= (uint32_t)tl.ntc;
    // the plane: direction i and the two transverse coordinates, the first
    // fastest (planes of neighbouring blocks share 32-byte sectors)
    const int q0 = (int)(b % (uint32_t)g.ns);
    b /= (uint32_t)g.ns;
    const int q1 = (int)(b % (uint32_t)g.ns);
    b /= (uint32_t)g.ns;
    const int x0 = (int)(b % (uint32_t)tl.nx) * tl.bx;
    b /= (uint32_t)tl.nx;
    const int t0 = (int)(b % (uint32_t)tl.nt) * tl.bt;
    const int i = (int)(b / (uint32_t)tl.nt);
    const int rcnt = FULL ? kLoopChunk : min(kLoopChunk, rmax - r0), tcnt = min(kLoopChunk, tmax - tc0);
    const TileSmem lay = tile_smem(tl.bx, tl.bt, rc, tl.tc, g.ns, r0);
    float4 *const s_ui = sm, *const s_ut = sm + lay.ut;
    float4 *const s_buf = sm + lay.s;  // [row t0 + tc0 + j][column][R]
    const int stride_i = g.stride[i];
    const int lex_plane = q0 * g.stride[i == 0 ? 1 : 0] + q1 * g.stride[i == 2 ? 1 : 2];
    const float4 *const Li = L + link_index(g, i, 0, 0);
    const float4 *const Lt = L + link_index(g, 3, 0, 0);
    auto link = [&](const float4 *dir, int a, int t) {  // 0 <= a < ns, 0 <= t < nt
        const int lex = t * g.vs + a * stride_i + lex_plane;
        const int parity = (a + t + q0 + q1) & 1;
        return __ldg(dir + (uint32_t)parity * (uint32_t)g.vh + (uint32_t)(lex >> 1));
    };

    for (int q = threadIdx.x; q < 2 * kLoopChunk * kLoopChunk; q += blockDim.x)
        s_sum[q] = 0u - blockDim.x * kSplitBits;
    for (int q = threadIdx.x; q < (tl.bt + tcnt) * lay.ucols; q += blockDim.x) {
        const int j = q / lay.ucols, d = q - j * lay.ucols;
        const int a = (x0 + d) % g.ns, t = (t0 + tc0 + j) % g.nt;
        s_ui[q] = link(Li, a, t);
        if (j < tl.bt + tcnt - 1) s_ut[q] = link(Lt, a, t);
    }
    __syncthreads();
    // S_R on the rows t0 + tc0 + j; d: the column's place in the staged row,
    // which wraps only when the row holds the whole extent
    for (int q = threadIdx.x; q < (tl.bt + tcnt) * tl.bx; q += blockDim.x) {
        const int j = q / tl.bx;
        const float4 *const u = s_ui + j * lay.ucols;
        float4 *const to = s_buf + q * tp;
        int d = q - j * tl.bx;
        float4 s = u[d];
        if (r0 == 0) to[0] = s;
        for (int r = 1; r < r0 + rcnt; ++r) {
            d = wrap_once(d + 1, lay.ucols);
            s = qmul(s, u[d]);
            if (r >= r0) to[r - r0] = s;
        }
    }
    // this thread's site: column c, row k of the tile; threads past the tile
    // and sites past the plane's edge compute on clamped indices and add zero
    // (their s_bot is zero)
    const int site = min((int)threadIdx.x, tl.bx * tl.bt - 1);
    const int k = site / tl.bx, c = site - k * tl.bx;
    const bool active = (int)threadIdx.x < tl.bx * tl.bt && x0 + c < g.ns && t0 + k < g.nt;
    // the column next to the tile that this thread extends: h < rcnt <= bx
    const int hk = (int)threadIdx.x / rcnt, h = (int)threadIdx.x - hk * rcnt;
    const bool halo = hk < tl.bt;
    // T_T at the site, at its column + r0, and at the halo column, after the
    // steps before this chunk (walked from global memory; none in the first)
    float4 tt0 = make_float4(1.0f, 0.0f, 0.0f, 0.0f), tb = tt0, th = tt0;
    float4 s_bot[kLoopChunk];
    __syncthreads();  // s_buf is complete, the staged U_i is done with
    if (tc0 == 0) {
#pragma unroll
        for (int r = 0; r < kLoopChunk; ++r) s_bot[r] = s_buf[site * tp + min(r, rcnt - 1)];
    } else {  // the site's own row is not among the staged ones
        int a = (x0 + c) % g.ns;
        const int t = (t0 + k) % g.nt;
        float4 s = link(Li, a, t);
        for (int r = 1; r <= r0; ++r) {
            a = wrap_once(a + 1, g.ns);
            s = qmul(s, link(Li, a, t));
        }
        s_bot[0] = s;
#pragma unroll
        for (int r = 1; r < kLoopChunk; ++r) {
            a = wrap_once(a + 1, g.ns);
            if (r < rcnt) s = qmul(s, link(Li, a, t));
            s_bot[r] = s;
        }
        auto walk = [&](int col, int row) {
            const int ca = col % g.ns;
            int ct = row % g.nt;
            float4 p = link(Lt, ca, ct);
            for (int step = 1; step < tc0; ++step) {
                ct = wrap_once(ct + 1, g.nt);
                p = qmul(p, link(Lt, ca, ct));
            }
            return p;
        };
        tt0 = walk(x0 + c, t0 + k);
        if (r0 > 0) tb = walk(x0 + c + r0, t0 + k);
        if (halo) th = walk(x0 + r0 + tl.bx + h, t0 + hk);
    }
    if (!active) {
#pragma unroll
        for (int r = 0; r < kLoopChunk; ++r) s_bot[r] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    const float4 *ut = s_ut + k * lay.ucols + c;
    const int tb_off = wrap_once(c + r0, lay.ucols) - c;
    const float4 *ut_h = s_ut + hk * lay.ucols + wrap_once(tl.bx + r0 + h, lay.ucols);
    float4 *own_to = sm + k * pitch + c, *halo_to = sm + hk * pitch + tl.bx + h;
    const float4 *top = s_buf + (site + tl.bx) * tp;  // the site one step of T above, then two ...

    const int lane = threadIdx.x & 31;
    bool outside = false;
    unsigned int acc_h = 0, acc_l = 0;  // lane (T & 3) 8 + R of the current four steps of T
    auto flush = [&](int tt_first) {
        const int idx = 2 * (tt_first * kLoopChunk + lane);
        atomicAdd(&s_sum[idx], acc_h);
        atomicAdd(&s_sum[idx + 1], acc_l);
        acc_h = acc_l = 0;
    };
    for (int tt = 0; tt < tcnt; ++tt) {
        const int flip = (tt & 1) * buf_len;
        const bool first = tc0 + tt == 0;  // block-uniform
        const float4 u = *ut;
        tt0 = first ? u : qmul(tt0, u);
        if (r0 > 0) {
            const float4 ub = ut[tb_off];
            tb = first ? ub : qmul(tb, ub);
        } else {
            tb = tt0;
        }
        if ((int)threadIdx.x < tl.bx * tl.bt) own_to[flip] = tb;
        if (halo) {
            const float4 uh = *ut_h;
            th = first ? uh : qmul(th, uh);
            halo_to[flip] = th;
        }
        ut += lay.ucols;
        ut_h += lay.ucols;
        __syncthreads();
        const float4 *const row = own_to + flip + 1;
        const int acc_r = lane - (tt & 3) * kLoopChunk;  // the R whose sums this lane takes
#pragma unroll
        for (int r = 0; r < kLoopChunk; ++r) {
            if (r < rcnt) {  // block-uniform
                const float4 A = qmul(s_bot[r], row[r]);
                const float4 B = qmul(tt0, top[r]);
                const float x = chain4(A.x, B.x, A.y, B.y, A.z, B.z, A.w, B.w);
                outside |= !(fabsf(x) < 2.0f);
                const float y = __fadd_rn(x, kSplit);
                const float z = __fmaf_rn(__fsub_rn(x, __fsub_rn(y, kSplit)), 0x1p22f, kSplit);
                const unsigned int hs = __reduce_add_sync(0xffffffffu, __float_as_uint(y));
                const unsigned int ls = __reduce_add_sync(0xffffffffu, __float_as_uint(z));
                if (acc_r == r) {
                    acc_h += hs;
                    acc_l += ls;
                }
            }
        }
        top += tl.bx * tp;
        if ((tt & 3) == 3) flush(tt - 3);
    }
    if (tcnt & 3) flush(tcnt & ~3);
    if (__any_sync(0xffffffffu, outside) && lane == 0) atomicOr(flag, 1u);
    __syncthreads();
    // the block's sums into its slot: [slot][R][T][h, l]
    unsigned long long *const slot = slots + (size_t)(blockIdx.x % (uint32_t)nslots) * (size_t)(2 * rmax * tmax);
    for (int q = threadIdx.x; q < kLoopChunk * tcnt; q += blockDim.x) {
        const int r = q & (kLoopChunk - 1), tt = q >> 3;
        if (r >= rcnt) continue;
        unsigned long long *const d = slot + 2 * ((r0 + r) * tmax + tc0 + tt);
        const int vh = (int)s_sum[2 * q], vl = (int)s_sum[2 * q + 1];
        if (vh) atomicAdd(d, (unsigned long long)(long long)vh);
        if (vl) atomicAdd(d + 1, (unsigned long long)(long long)vl);
    }
}

// out[o] = scale (sum over slots), one warp per output; out[n_out] = the flag.
__global__ void wilson_tile_finish_kernel(const unsigned long long *__restrict__ slots, int nslots, int n_out,
                                          double scale, const unsigned int *__restrict__ flag,
                                          double *__restrict__ out)
{
    const int o = blockIdx.x;
    long long h = 0, l = 0;
    for (int s = threadIdx.x; s < nslots; s += 32) {
        h += (long long)slots[((size_t)s * n_out + o) * 2];
        l += (long long)slots[((size_t)s * n_out + o) * 2 + 1];
    }
    for (int off = 16; off > 0; off >>= 1) {
        h += __shfl_down_sync(0xffffffffu, h, off);
        l += __shfl_down_sync(0xffffffffu, l, off);
    }
    if (threadIdx.x == 0) {
        out[o] = ((double)h * 0x1p-21 + (double)l * 0x1p-43) * scale;
        if (o == 0) out[n_out] = *flag ? 1.0 : 0.0;
    }
}

// ------------------------------------------------------ binary64 kernel
// One launch per T: each thread takes (site, direction) items and, for R = 1
// .. rmax, extends S_R and the line at height T by one link and walks
// T_T(x+Ri); per-R binary64 sums in registers, block partials in a fixed
// order.  The faster one for few small loops (walks_are_faster), and as it takes
// any links it finishes the calls whose loops the tiled kernel's fixed point
// does not hold (24^4 up to 8 x 8: 1.2 ms).
struct Site {
    int c[4];
};

__device__ __forceinline__ float4 link_at_site(const float4 *__restrict__ L, const Geom &g, const Site &s, int mu)
{
    const int lex = ((s.c[3] * g.ns + s.c[2]) * g.ns + s.c[1]) * g.ns + s.c[0];
    const int parity = (s.c[0] + s.c[1] + s.c[2] + s.c[3]) & 1;
    return __ldg(L + link_index(g, mu, parity, lex >> 1));
}

__device__ __forceinline__ void step(const Geom &g, Site &s, int mu)
{
    const int c = s.c[mu] + 1;
    s.c[mu] = c == g.ext[mu] ? 0 : c;
}

template <int RM>
__global__ void __launch_bounds__(kWilsonThreads) wilson_kernel(const float4 *__restrict__ L, Geom g, int rmax, int T,
                                                                double *__restrict__ partials)
{
    double acc[RM];
#pragma unroll
    for (int r = 0; r < RM; ++r) acc[r] = 0.0;
    const int64_t items = 6 * (int64_t)g.vh;  // 3 V
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < items;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int site = (int)(q / 3);
        const int i = (int)(q - 3 * (int64_t)site);
        Site x;
        {
            const uint32_t rest = fastdiv((uint32_t)site, g.div_ns);
            x.c[0] = site - (int)rest * g.ns;
            const uint32_t rest2 = fastdiv(rest, g.div_ns);
            x.c[1] = (int)rest - (int)rest2 * g.ns;
            x.c[3] = (int)fastdiv(rest2, g.div_ns);
            x.c[2] = (int)rest2 - x.c[3] * g.ns;
        }
        // T_T(x) and the corner x + T t
        Site xt = x;
        float4 tt0 = link_at_site(L, g, xt, 3);
        step(g, xt, 3);
        for (int j = 1; j < T; ++j) {
            tt0 = qmul(tt0, link_at_site(L, g, xt, 3));
            step(g, xt, 3);
        }
        Site xs = x;  // x + (R-1) i along the bottom, then x + R i
        Site ys = xt; // x + T t + (R-1) i along the top
        float4 s_bot = make_float4(1.0f, 0.0f, 0.0f, 0.0f), s_top = s_bot;
#pragma unroll
        for (int r = 0; r < RM; ++r) {
            if (r < rmax) {
                const float4 ub = link_at_site(L, g, xs, i);
                const float4 ut = link_at_site(L, g, ys, i);
                s_bot = r == 0 ? ub : qmul(s_bot, ub);
                s_top = r == 0 ? ut : qmul(s_top, ut);
                step(g, xs, i);
                step(g, ys, i);
                // T_T(x + (r+1) i)
                Site z = xs;
                float4 tt = link_at_site(L, g, z, 3);
                step(g, z, 3);
                for (int j = 1; j < T; ++j) {
                    tt = qmul(tt, link_at_site(L, g, z, 3));
                    step(g, z, 3);
                }
                const float4 a = qmul(s_bot, tt);
                const float4 b = qmul(tt0, s_top);
                acc[r] += (double)chain4(a.x, b.x, a.y, b.y, a.z, b.z, a.w, b.w);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < RM; ++r) {
        const double v = block_sum(acc[r]);
        if (threadIdx.x == 0 && r < rmax) partials[(size_t)blockIdx.x * rmax + r] = v;
    }
}

// out[(R-1) tmax + (T-1)] = (sum over blocks, in order) / (3 V) for R = 1 .. rmax.
__global__ void wilson_finish_kernel(const double *__restrict__ partials, int nblocks, int rmax, int T, int tmax,
                                     double scale, double *__restrict__ out)
{
    for (int r = 0; r < rmax; ++r) {
        double v = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += blockDim.x) v += partials[(size_t)b * rmax + r];
        v = block_sum(v);
        if (threadIdx.x == 0) out[r * tmax + (T - 1)] = v * scale;
    }
}

// Enqueues the walks; the values go to the reduction scratch, behind the
// block partials.  *d_out: their device address.
template <int RM>
static cudaError_t launch_wilson(su2_lattice *lat, int rmax, int tmax, double **d_out)
{
    const Geom g = geom_of(lat);
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, lat->device);
    const int room = (lat->scratch.partials_cap - rmax * tmax) / rmax;
    const int grid = grid_for(6 * (int64_t)g.vh, kWilsonThreads, std::min(4 * sms, room));
    const double scale = 1.0 / (6.0 * (double)g.vh);
    *d_out = lat->scratch.partials + (size_t)grid * rmax;
    for (int T = 1; T <= tmax; ++T) {
        wilson_kernel<RM><<<grid, kWilsonThreads, 0, lat->stream>>>(lat->links, g, rmax, T, lat->scratch.partials);
        wilson_finish_kernel<<<1, kWilsonThreads, 0, lat->stream>>>(lat->scratch.partials, grid, rmax, T, tmax,
                                                                   scale, *d_out);
    }
    return cudaGetLastError();
}

static cudaError_t launch_walks(su2_lattice *lat, int rmax, int tmax, double **d_out)
{
    return rmax <= 4   ? launch_wilson<4>(lat, rmax, tmax, d_out)
           : rmax <= 8 ? launch_wilson<8>(lat, rmax, tmax, d_out)
                       : launch_wilson<16>(lat, rmax, tmax, d_out);
}

// The tiles of a call: whole rows (more than 64 columns in even parts) and as
// many time slices as fit 256 threads, in even tiles.
static LoopTiles loop_tiles(int ns, int nt, int rmax, int tmax)
{
    LoopTiles tl;
    tl.nx = (ns + kTileMaxBx - 1) / kTileMaxBx;
    tl.bx = (ns + tl.nx - 1) / tl.nx;
    tl.bt = std::min(nt, std::max(1, kTileThreads / tl.bx));
    tl.nt = (nt + tl.bt - 1) / tl.bt;
    tl.bt = (nt + tl.nt - 1) / tl.nt;
    tl.rc = std::min(rmax, kLoopChunk);
    tl.tc = std::min(tmax, kLoopChunk);
    tl.nr = (rmax + kLoopChunk - 1) / kLoopChunk;
    tl.ntc = (tmax + kLoopChunk - 1) / kLoopChunk;
    return tl;
}

static int tile_threads(const LoopTiles &tl) { return std::max(32, (tl.bx * tl.bt + 31) & ~31); }

// The walks load, per site and direction, T links of the line at the site and
// for each R one of S_R, one of its top and T of the far line: `loads` for all
// extents, at about 3 ps each (48^4) and 13 us per launch (one per T).  A tile
// costs 14 to 15 such loads per chunk before its first loop, over the threads
// that its sites leave idle (more on a large lattice, less on one that stays
// in L2), and little per loop after it.  So the walks stay the faster ones for
// few small loops, from about 20^4 on (16^4, 3 x 1: 41 / 36).  us per call on
// the walks / the tiles:
//   R x T        1 x 1       2 x 1       4 x 1       2 x 2       4 x 2       8 x 1
//   24^4       43 / 68     54 / 69     68 / 72     94 / 74    132 / 85    116 / 82
//   48^4     217 / 728   352 / 790   658 / 900   753 / 936 1417 / 1099  1325 / 947
static bool walks_are_faster(const su2_lattice *lat, int rmax, int tmax)
{
    const LoopTiles tl = loop_tiles(lat->ns, lat->nt, rmax, tmax);
    const double vol = (double)lat->vol, chunks = tl.nr * tl.ntc;
    const double loads = 0.5 * tmax * (tmax + 1) * (1 + rmax) + 2.0 * tmax * rmax;
    const double filled = (double)lat->ns * lat->nt / ((double)tl.nx * tl.nt * tile_threads(tl));
    const double most = vol < 1e6 ? 14.0 : chunks == 1.0 ? 22.0 : 18.0 * chunks;
    return loads * filled <= most && vol >= 1e5 + 3e5 * (tmax - 1);
}

// Enqueues the tiled kernel.  The sums live in the reduction scratch, in as many slots as fit (blocks spread over
// the slots, so their atomics meet rarely), the results behind them: rmax tmax
// values and the flag.  *d_out: their device address.
static cudaError_t launch_tiles(su2_lattice *lat, int rmax, int tmax, double **d_out)
{
    const Geom g = geom_of(lat);
    const int n_out = rmax * tmax;
    const LoopTiles tl = loop_tiles(g.ns, lat->nt, rmax, tmax);
    const int nslots = std::min(256, (lat->scratch.partials_cap - n_out - 2) / (2 * n_out));
    unsigned long long *slots = (unsigned long long *)lat->scratch.partials;
    unsigned int *flag = (unsigned int *)(slots + (size_t)nslots * 2 * n_out);
    *d_out = (double *)(flag + 2);
    cudaError_t e = cudaMemsetAsync(slots, 0, sizeof(double) * ((size_t)nslots * 2 * n_out + 1), lat->stream);
    if (e != cudaSuccess) return e;
    const size_t smem = sizeof(float4) * (size_t)tile_smem(tl.bx, tl.bt, tl.rc, tl.tc, g.ns, (tl.nr - 1) * kLoopChunk).total;
    const auto kernel = rmax % kLoopChunk == 0 ? wilson_tile_kernel<true> : wilson_tile_kernel<false>;
    // the limit belongs to the kernel, which other threads launch too: always the most that a tile takes
    e = smem <= kTileMaxSmem ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileMaxSmem)
                             : cudaErrorInvalidValue;
    if (e != cudaSuccess) return e;
    const unsigned int blocks = 3u * (unsigned int)(g.ns * g.ns) * (unsigned int)(tl.nx * tl.nt * tl.nr * tl.ntc);
    kernel<<<blocks, tile_threads(tl), smem, lat->stream>>>(lat->links, g, tl, rmax, tmax, slots, nslots, flag);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    wilson_tile_finish_kernel<<<n_out, 32, 0, lat->stream>>>(slots, nslots, n_out, 1.0 / (6.0 * (double)g.vh), flag,
                                                             *d_out);
    return cudaGetLastError();
}

}  // namespace su2

using namespace su2;

extern "C" su2_status su2_wilson_loops(su2_lattice *lat, int rmax, int tmax, double *out)
{
    if (!lat || !out || rmax < 1 || tmax < 1 || rmax > kWilsonMaxR || tmax > kWilsonMaxT || rmax > lat->ns ||
        tmax > lat->nt) {
        set_last_error("su2_wilson_loops: 1 <= rmax <= min(16, Ns), 1 <= tmax <= min(64, Nt), out != NULL");
        return SU2_E_INVAL;
    }
    DeviceGuard guard(lat->device);
    const size_t n_out = (size_t)rmax * (size_t)tmax;
    HostPage page(lat->stream);
    double own[kWilsonMaxR * kWilsonMaxT + 1];
    double *const host = page.p ? (double *)page.p : own;
    double *d_out = nullptr;
    bool walk = walks_are_faster(lat, rmax, tmax);
    for (;;) {
        SU2_CUDA(walk ? launch_walks(lat, rmax, tmax, &d_out) : launch_tiles(lat, rmax, tmax, &d_out));
        const size_t n = walk ? n_out : n_out + 1;  // the tiles' values are followed by their flag
        SU2_CUDA(cudaMemcpyAsync(host, d_out, sizeof(double) * n, cudaMemcpyDeviceToHost, lat->stream));
        SU2_CUDA(cudaStreamSynchronize(lat->stream));
        if (walk || host[n_out] == 0.0) break;
        walk = true;  // a loop outside (-2, 2)
    }
    page.settled();
    std::copy(host, host + n_out, out);
    return SU2_OK;
}
