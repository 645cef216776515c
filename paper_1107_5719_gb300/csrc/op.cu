// The recorded formal solution as an assembled operator.
//
// With the opacities, directions and boundary values fixed, the formal
// solution is linear in the source S (Hauschildt & Baron 2011, Sect. 2.2: I is
// a weighted sum of S along the characteristic plus the transmitted boundary
// intensity).  Because voxel centres are lattice points, the upstream points
// of a direction touch the same node offsets for every voxel of a plane, so
// the contributions of all directions to one node offset add up to one
// coefficient per voxel:
//   J_v = c0_v S_v + bc_v + sum_e A[e][v] S[v + off_e],
// the offsets e of plane k0 being, for each sign of mu and each distance m,
// the distinct nodes the directions of that sign touch m planes away.  Per
// replayed step (four nodes) the 65^3 slab with 32 x 32 directions holds 2.2
// distinct nodes, so a formal solution is 2.2 FP64 operations per step
// instead of the five of interpolating S at every step, and 8 bytes of
// coefficient per operation.
//
// Recording, once per opacity:
//   k_op_lists   (once per quadrature) per (sign, distance) the distinct
//                nodes, the steepest directions' first (they are cut off
//                last, so the nodes still in use are a prefix), and per node
//                its contributions (direction, w_d times the bilinear weight)
//   k_op_len     the length of every warp's rays, from an FP32 march
//   k_op_counts  per (plane, sign, distance) the prefix of nodes in use
//   k_rec64      the march's coefficients c_m of S(p_m) of one chunk of planes
//   k_op_assemble  A[e][v] = sum over e's contributions of w_d b c_m
// and k_op_apply64 evaluates J for a source.
#include "df.cuh"
#include "internal.h"
#include "weights.cuh"

#include <cooperative_groups.h>

namespace rt3d {

namespace {
namespace cg = cooperative_groups;

constexpr int kOpThreads = 128;      // march and length kernels
constexpr int kListThreads = 256;

struct OpNodes {
    int a00, a10, a01, a11;
};

__device__ __forceinline__ OpNodes op_nodes(int i0, int j0, int ox, int oy, int nx, int ny)
{
    int x0 = i0 + ox;
    x0 -= x0 >= nx ? nx : 0;
    const int x1 = x0 + 1 == nx ? 0 : x0 + 1;
    int y0 = j0 + oy;
    y0 -= y0 >= ny ? ny : 0;
    const int y1 = y0 + 1 == ny ? 0 : y0 + 1;
    return OpNodes{y0 * nx + x0, y0 * nx + x1, y1 * nx + x0, y1 * nx + x1};
}

__device__ __forceinline__ int op_nmax(OpNodes n) { return max(max(n.a00, n.a10), max(n.a01, n.a11)); }
__device__ __forceinline__ int op_nmin(OpNodes n) { return min(min(n.a00, n.a10), min(n.a01, n.a11)); }

__device__ __forceinline__ double op_bilin(const double* __restrict__ p, OpNodes n, Bw4d b)
{
    return b.x * __ldg(p + n.a00) + b.y * __ldg(p + n.a10) + b.z * __ldg(p + n.a01) +
           b.w * __ldg(p + n.a11);
}

// One block per (sign, slot m): the distinct nodes of the directions of that
// sign at distance m (m >= 1), or at the downstream point (m = 0, when dn is
// given), in the order of the direction list (decreasing |mu|); then each
// node's contributions in the same order.  Item i of the block is corner
// i & 3 of direction dl[i >> 2].
__global__ void __launch_bounds__(kListThreads)
k_op_lists(Geometry g, const DirInfo* __restrict__ info, const StepGeo* __restrict__ off,
           const Bw4d* __restrict__ bw, const DownGeo* __restrict__ dn, OpLists L, int* gfirst)
{
    extern __shared__ int sfirst[];
    __shared__ int wsum[kListThreads / 32];
    const int nx = g.nx, ny = g.ny, nz = g.nz, nxy = nx * ny;
    const int si = blockIdx.x / nz, m = blockIdx.x - si * nz;
    const int D = si == 0 ? L.dpos : g.ndir - L.dpos;
    const int* dl = L.dord + (si == 0 ? 0 : L.dpos);
    const long long row = (long long)si * nz + m;
    const int n = (m == 0 && !dn) ? 0 : 4 * D;
    int* first = gfirst ? gfirst + row * nxy : sfirst;
    int* unode = L.unode + row * L.ucap;
    int* ustart = L.ustart + row * (L.ucap + 1);
    int* uofi = L.uofi + row * L.icap;
    OpContrib* ct = L.contrib + row * L.icap;
    auto node = [&](int i) {
        const int d = dl[i >> 2];
        int x, y;
        if (m == 0) {
            x = dn[d].ox;
            y = dn[d].oy;
        } else {
            const StepGeo o = off[(long long)d * nz + m];
            x = o.ox;
            y = o.oy;
        }
        x += i & 1;
        x -= x == nx ? nx : 0;
        y += (i >> 1) & 1;
        y -= y == ny ? ny : 0;
        return y * nx + x;
    };
    for (int t = threadIdx.x; t < nxy; t += kListThreads) first[t] = 0x7fffffff;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kListThreads) atomicMin(&first[node(i)], i);
    __syncthreads();
    // ordered compaction of the items that are the first of their node; a
    // node's entry then holds -(position + 1)
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int base = 0;
    for (int i0 = 0; i0 < n; i0 += kListThreads) {
        const int i = i0 + threadIdx.x;
        const int nd = i < n ? node(i) : 0;
        const bool f = i < n && first[nd] == i;
        const unsigned b = __ballot_sync(0xffffffffu, f);
        if (lane == 0) wsum[wid] = __popc(b);
        __syncthreads();
        int pre = base, tot = 0;
        for (int w = 0; w < kListThreads / 32; ++w) {
            if (w < wid) pre += wsum[w];
            tot += wsum[w];
        }
        if (f) {
            const int pos = pre + __popc(b & ((1u << lane) - 1));
            first[nd] = -(pos + 1);
            unode[pos] = nd;
        }
        base += tot;
        __syncthreads();
    }
    const int U = base;
    for (int i = threadIdx.x; i < n; i += kListThreads) uofi[i] = -first[node(i)] - 1;
    // where the 27-point neighbourhood's nodes are in the list (m <= 1)
    if (m <= 1 && threadIdx.x < 9) {
        const int ox = threadIdx.x % 3 - 1, oy = threadIdx.x / 3 - 1;
        const int f = n ? first[(oy < 0 ? ny - 1 : oy) * nx + (ox < 0 ? nx - 1 : ox)] : 0;
        L.lpos[(si * 2 + m) * 9 + threadIdx.x] = f < 0 ? -f - 1 : -1;
    }
    __syncthreads();
    // the prefix of the list that direction d needs
    for (int q = threadIdx.x; 4 * q < n; q += kListThreads) {
        const int* u = uofi + 4 * q;
        L.posmax[(long long)dl[q] * nz + m] = max(max(u[0], u[1]), max(u[2], u[3])) + 1;
    }
    __syncthreads();
    // contributions: counts, their prefix sums, then the entries in item order (in
    // time linear in the items; every thread looking through all items for its
    // nodes took 3.4 ms for 33 planes of 4096 directions, and the first formal
    // solution after a quadrature in double-float 32.4 ms against 29.4)
    int* next = first;           // its nodes are looked up
    for (int u = threadIdx.x; u < U; u += kListThreads) next[u] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kListThreads) atomicAdd(&next[uofi[i]], 1);
    __syncthreads();
    base = 0;
    for (int u0 = 0; u0 < U; u0 += kListThreads) {
        const int u = u0 + threadIdx.x, v = u < U ? next[u] : 0;
        int x = v;
        for (int h = 1; h < 32; h <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, h);
            if (lane >= h) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        int pre = base, tot = 0;
        for (int w = 0; w < kListThreads / 32; ++w) {
            if (w < wid) pre += wsum[w];
            tot += wsum[w];
        }
        if (u < U) {
            ustart[u] = next[u] = pre + x - v;
            if (u == U - 1) ustart[U] = pre + x;
        }
        base += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        L.ucount[row] = U;
        if (U == 0) ustart[0] = 0;
    }
    // the places, 32 items at a time: an item comes after those of its node in
    // lower lanes and in earlier rounds
    if (wid == 0)
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane, u = i < n ? uofi[i] : -1;
            const unsigned same = __match_any_sync(0xffffffffu, u);
            const int j = u < 0 ? 0 : next[u] + __popc(same & ((1u << lane) - 1));
            __syncwarp();
            if (u >= 0) {
                if (lane == __ffs(same) - 1) next[u] += __popc(same);
                ct[j].d = i;
                ct[j].ul = 2 * u + (j == ustart[u + 1] - 1);
            }
            __syncwarp();
        }
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += kListThreads) {
        const int i = ct[j].d, d = dl[i >> 2], q = i & 3;
        const Bw4d b = m == 0 ? dn[d].b : bw[(long long)d * nz + m];
        ct[j].wb = info[d].w * (q == 0 ? b.x : q == 1 ? b.y : q == 2 ? b.z : b.w);
        ct[j].d = d;
    }
}

// 1 / smax (0 for a source that is zero everywhere)
__device__ __forceinline__ double over_smax(const double* __restrict__ smax)
{
    const double sm = *smax;
    return sm > 0.0 ? 1.0 / sm : 0.0;
}

// node2[k][y][x] = {chi, S / smax} in FP32 (OWN: {chi, chi of the next x}, all
// that the march of k_op_len<OWN> reads, in half its loads), planes padded to
// 2ny x 2nx by periodic copies.  chi is kept below 1e25 (opaque in any case)
// so that the FP32 march forms no infinities.
template <bool OWN>
__global__ void k_op_pack_len(Geometry g, const double* __restrict__ chi,
                              const double* __restrict__ S, const double* __restrict__ smax,
                              float2* __restrict__ node)
{
    const int nx = g.nx, ny = g.ny;
    const long long W = 2LL * nx, P = 4LL * nx * ny;
    const double inv = OWN ? 0.0 : over_smax(smax);
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < g.N;
         v += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(v % nx), j = (int)((v / nx) % ny);
        const long long k = v / ((long long)nx * ny);
        const float c = (float)fmin(chi[v], 1e25);
        const float2 q = OWN ? make_float2(c, (float)fmin(chi[i + 1 == nx ? v - i : v + 1], 1e25))
                             : make_float2(c, (float)(S[v] * inv));
        float2* p = node + k * P + (long long)j * W + i;
        p[0] = q;
        p[nx] = q;
        p[(long long)ny * W] = q;
        p[(long long)ny * W + nx] = q;
    }
}

// Lengths of the rays, from a march in FP32.  A ray ends once the rest of it
// can change I by less than 2^-lcut |I|, i.e. T smax <= 2^-lcut |I| (tested
// on logarithms: tau log2 e + log2(|I| / smax) >= lcut); OWN (double-float):
// by less than 2^-lcut of the voxel's own source, which takes no intensity, and
// two pairs of opacities a step in place of four nodes (38 x 46 x 36 with 198
// directions: 213 -> 171 us).  The 32 lanes of a warp share the longest of their
// rays.
template <bool OWN>
__global__ void __launch_bounds__(kOpThreads)
k_op_len(Geometry g, const float2* __restrict__ node, const double* __restrict__ S,
         const double* __restrict__ smax, const DirInfo* __restrict__ info,
         const int* __restrict__ poff, const float4* __restrict__ bw, float lcut,
         int* __restrict__ lmax, int nwp)
{
    constexpr float kLog2e = 1.4426950408889634f;
    const int nx = g.nx, nz = g.nz, nxy = nx * g.ny;
    const int t = blockIdx.x * kOpThreads + threadIdx.x;
    const int k0 = plane_at(g, blockIdx.z);
    const bool active = t < nxy;
    const unsigned amask = __ballot_sync(0xffffffffu, active);
    if (!active) return;
    const int j0 = t / nx, i0 = t - j0 * nx;
    const long long W = 2LL * nx, P = 4LL * nxy;
    const long long base = k0 * P + j0 * W + i0;
    float2 me = node[base];
    if (OWN) me.y = (float)(S[(long long)k0 * nxy + t] * over_smax(smax));
    const float2* nb = node + base;
    float own;      // NaN for S < 0, -inf for S = 0: never cut
    asm("lg2.approx.f32 %0, %1;" : "=f"(own) : "f"(me.y));
    for (int d = blockIdx.y; d < g.ndir; d += gridDim.y) {
        const int s = info[d].sgn;
        const float hs = info[d].hs32;
        const int M = s > 0 ? k0 : nz - 1 - k0;
        const int* od = poff + (long long)d * nz;
        const float4* bd = bw + (long long)d * nz;
        float I = 0.f, T = 1.f, tau = 0.f, ca = me.x, sa = me.y;
        int m = 0;
        while (m < M) {
            const int o = od[m + 1];
            RT_GUARD(g, base + o, 4 * g.N, kSiteFs64) break;
            RT_GUARD(g, base + o + W + 1, 4 * g.N, kSiteFs64) break;
            const float4 b = bd[m + 1];
            const float2* q = nb + o;
            float2 q00 = __ldg(q), q01 = __ldg(q + W), q10, q11;
            if (OWN) {
                q10 = make_float2(q00.y, 0.f);
                q11 = make_float2(q01.y, 0.f);
            } else {
                q10 = __ldg(q + 1);
                q11 = __ldg(q + W + 1);
            }
            const float cb = b.x * q00.x + b.y * q10.x + b.z * q01.x + b.w * q11.x;
            const float x = hs * (ca + cb);
            float lg = own;
            if (!OWN) {
                const float sb = b.x * q00.y + b.y * q10.y + b.z * q01.y + b.w * q11.y;
                float wc, wu, e;
                seg_weights32(x, wc, wu, e);
                I = fmaf(T, fmaf(wc, sa, wu * sb), I);
                sa = sb;
                asm("lg2.approx.f32 %0, %1;" : "=f"(lg) : "f"(fabsf(I)));
            }
            tau += x;
            if (!OWN) T = ex2_approx(-tau * kLog2e);
            ca = cb;
            ++m;
            if (fmaf(tau, kLog2e, lg) >= lcut) break;
        }
        const int Lw = __reduce_max_sync(amask, m);
        if ((threadIdx.x & 31) == 0) lmax[((long long)d * nz + k0) * nwp + (t >> 5)] = Lw;
    }
}

// Per (plane k0, direction d): the longest warp, Lp; and the voxel-steps of
// all of them into *steps.  One warp per (k0, d).
__global__ void k_op_plane_len(Geometry g, const int* __restrict__ lmax, int nwp,
                               int* __restrict__ Lp, unsigned long long* __restrict__ steps)
{
    const int lane = threadIdx.x & 31;
    const int d = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), k0 = blockIdx.y;
    if (d >= g.ndir) return;
    const int last = g.nx * g.ny - 32 * (nwp - 1);      // lanes of the plane's last warp
    int L = 0;
    unsigned long long s = 0;
    for (int w = lane; w < nwp; w += 32) {
        const int l = lmax[((long long)d * g.nz + k0) * nwp + w];
        L = max(L, l);
        s += (unsigned long long)l * (w == nwp - 1 ? last : 32);
    }
    L = __reduce_max_sync(0xffffffffu, L);
    for (int h = 16; h > 0; h >>= 1) s += __shfl_down_sync(0xffffffffu, s, h);
    if (lane == 0) {
        Lp[(long long)k0 * g.ndir + d] = L;
        if (s) atomicAdd(steps, s);
    }
}

// Per plane k0 (one block): the rows of the chunk buffer (row of (d, m) is
// rowbase[k0][d] + m - 1, with one more row first for the downstream point
// of the parabolic source), the entries per (sign, slot) rounded up to
// pairs, their first entry and the plane's number of entries, rounded up to
// kOpPad.
__global__ void __launch_bounds__(kListThreads)
k_op_counts(Geometry g, OpLists L, int para, const int* __restrict__ Lp, int* __restrict__ rowbase,
            int* __restrict__ cnt, int* __restrict__ segb, int* __restrict__ E, int* __restrict__ rows)
{
    __shared__ int wsum[kListThreads / 32];
    const int nz = g.nz, k0 = blockIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int* lp = Lp + (long long)k0 * g.ndir;
    int base = 0;
    for (int d0 = 0; d0 < g.ndir; d0 += kListThreads) {
        const int d = d0 + threadIdx.x;
        const int v = d < g.ndir ? lp[d] + para : 0;
        int x = v;
        for (int h = 1; h < 32; h <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, h);
            if (lane >= h) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        int pre = base, tot = 0;
        for (int w = 0; w < kListThreads / 32; ++w) {
            if (w < wid) pre += wsum[w];
            tot += wsum[w];
        }
        if (d < g.ndir) rowbase[(long long)k0 * g.ndir + d] = pre + x - v;
        base += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) rows[k0] = base;
    // a warp per (sign, distance), its lanes the directions; then a scan by
    // warp 0 (38 x 46 x 36 with 198 directions: 11.6 us, 25.5 with one thread to
    // each and a serial scan)
    int* cn = cnt + (long long)k0 * 2 * nz;
    for (int q = wid; q < 2 * nz; q += kListThreads / 32) {
        const int si = q / nz, m = q - si * nz, s = si ? -1 : 1;
        int n = 0;
        if (m == 0) {
            if (para && k0 + s >= 0 && k0 + s < nz) n = L.ucount[q];
        } else if (m <= (s > 0 ? k0 : nz - 1 - k0)) {
            const int D = si == 0 ? L.dpos : g.ndir - L.dpos;
            const int* dl = L.dord + (si == 0 ? 0 : L.dpos);
            for (int i = lane; i < D; i += 32)
                if (lp[dl[i]] >= m) n = max(n, L.posmax[(long long)dl[i] * nz + m]);
        }
        n = __reduce_max_sync(0xffffffffu, n);
        if (lane == 0) cn[q] = n;
    }
    __syncthreads();
    if (wid) return;
    int e = 0;
    for (int q0 = 0; q0 < 2 * nz; q0 += 32) {
        const int q = q0 + lane, v = q < 2 * nz ? (cn[q] + 1) & ~1 : 0;
        int x = v;
        for (int h = 1; h < 32; h <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, h);
            if (lane >= h) x += y;
        }
        if (q < 2 * nz) segb[(long long)k0 * 2 * nz + q] = e + x - v;
        e += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) E[k0] = (e + kOpPad - 1) / kOpPad * kOpPad;
}

// off[e]: the entry's node relative to the voxel in planes padded to
// 2ny x 2nx (0 for the padding entries, whose coefficients are 0).
__global__ void k_op_offsets(Geometry g, OpLists L, const int* __restrict__ cnt,
                             const int* __restrict__ segb, const int* __restrict__ E,
                             const long long* __restrict__ eb, int* __restrict__ off)
{
    const int nx = g.nx, nz = g.nz, k0 = blockIdx.y;
    int* o = off + eb[k0];
    for (int q = blockIdx.x; q <= 2 * nz; q += gridDim.x) {
        if (q == 2 * nz) {          // the plane's tail
            const int* sb = segb + (long long)k0 * 2 * nz;
            const int last = sb[2 * nz - 1] + ((cnt[(long long)k0 * 2 * nz + 2 * nz - 1] + 1) & ~1);
            for (int e = last + threadIdx.x; e < E[k0]; e += blockDim.x) o[e] = 0;
            continue;
        }
        const int si = q / nz, m = q - si * nz, s = si ? -1 : 1;
        const int n = cnt[(long long)k0 * 2 * nz + q], b = segb[(long long)k0 * 2 * nz + q];
        const long long dk = m == 0 ? s : -(long long)m * s;
        for (int u = threadIdx.x; u < ((n + 1) & ~1); u += blockDim.x) {
            int v = 0;
            if (u < n) {
                const int nd = L.unode[(long long)q * L.ucap + u], y = nd / nx, x = nd - y * nx;
                v = (int)((dk * 2 * g.ny + y) * 2 * nx + x);
            }
            o[b + u] = v;
        }
    }
}

// The march of the planes of rank r0 + blockIdx.z, its coefficients of S
// recorded: c_m = T_{m-1} w_up,{m-1} + T_m w_cur,m at row (d, m) (the last
// point: T_{L-1} w_up), and per voxel and slot sum_d w_d w_cur,0 and
// sum_d w_d T_L I_bc (rays that reach the boundary plane).  The lengths are
// given (k_op_len), so the march carries no intensity, no source and no
// cutoff test: about 21 FP64 instructions per step of the march that
// also forms I (the FP64 pipe bounds both).
__global__ void __launch_bounds__(kOpThreads)
k_rec64(Geometry g, int r0, const double* __restrict__ chi, const double* __restrict__ B,
        const double* __restrict__ G, const DirInfo* __restrict__ info,
        const StepGeo* __restrict__ off, const Bw4d* __restrict__ bw, const Bw4d* __restrict__ bwh,
        RecOut ro, const int* __restrict__ lmax, int nwp, double* __restrict__ c0s,
        double* __restrict__ bcs)
{
    const int nx = g.nx, ny = g.ny, nz = g.nz, nxy = nx * ny;
    const int t = blockIdx.x * kOpThreads + threadIdx.x;
    const int k0 = plane_at(g, r0 + blockIdx.z), zb = blockIdx.y, ZB = gridDim.y;
    __shared__ double tab[kExpTable];
    fill_exp_table(tab);
    __syncthreads();
    if (t >= nxy) return;
    const int j0 = t / nx, i0 = t - j0 * nx;
    const long long v = (long long)k0 * nxy + t;
    const double chi0 = chi[v];
    for (int slot = zb; slot < kSlots; slot += ZB) {
        double C0 = 0.0, Bc = 0.0;
        for (int d = slot; d < g.ndir; d += kSlots) {
            const int s = info[d].sgn;
            const double w = info[d].w;
            const int M = s > 0 ? k0 : nz - 1 - k0;
            const int L = lmax[((long long)d * nz + k0) * nwp + (t >> 5)];
            const StepGeo* od = off + (long long)d * nz;
            const Bw4d* bh = bwh + (long long)d * nz;
            double* rc = rec_rows(g, ro, ro.base, d, k0, s) + t;
            double T = 1.0, ca = info[d].hs * chi0, cprev = 0.0;
            for (int m = 0; m < L; ++m) {
                const long long pb = (long long)(k0 - (m + 1) * s) * nxy;
                const StepGeo o = od[m + 1];
                const OpNodes n = op_nodes(i0, j0, o.ox, o.oy, nx, ny);
                RT_GUARD(g, pb + op_nmin(n), g.N, kSiteFs64) break;
                RT_GUARD(g, pb + op_nmax(n), g.N, kSiteFs64) break;
                const double cb = op_bilin(chi + pb, n, bh[m + 1]);
                double b;
                const double before = cprev;
                seg_step64(T, ca + cb, tab, b, cprev, T);
                if (m == 0) C0 = fma(w, b, C0);
                else rc[(long long)(m - 1) * nxy] = before + b;
                ca = cb;
            }
            if (L > 0) rc[(long long)(L - 1) * nxy] = cprev;
            const int bc = s > 0 ? g.top_bc : g.bottom_bc;
            if (bc && L == M) {
                const long long pb = (long long)(k0 - M * s) * nxy;
                const StepGeo o = od[M];
                const OpNodes n = op_nodes(i0, j0, o.ox, o.oy, nx, ny);
                const Bw4d b = bw[(long long)d * nz + M];
                double ibc = op_bilin(B + pb, n, b);
                if (bc == 2) ibc = fma(info[d].amu, op_bilin(G, n, b), ibc);   // B + |mu| dB/dtau
                Bc = fma(w, T * ibc, Bc);
            }
        }
        c0s[(long long)slot * g.N + v] = C0;
        bcs[(long long)slot * g.N + v] = Bc;
    }
}

// A of the planes of rank r0 + blockIdx.y: one block per 32 voxels, the
// lanes of its warps the voxels.  A warp takes a run of entries of a list and
// walks their contributions, which are consecutive: 32 at a time, each lane
// looks one up and leaves its weight, row and entry in shared memory, then the
// warp adds them eight by eight in list order (eight coefficient loads in
// flight) and stores an entry when its last contribution is in.  Rows past the
// warp's own rays hold nothing (m > its length) and count as zero.
// FP64: bound by the FP64 pipe (81% busy; 33^3 with 256 directions 0.66 ms).  With
// the contributions passed by shuffles and the entries stored in pairs it took
// 2.5 times the instructions (0.74 ms; double-float 0.77 against 0.50).
constexpr int kAsmRun = 32;      // entries of a run (even)
constexpr int kAsmShared = 8 * 24 * 1024;    // the lengths of 24 Ki directions

// The two arithmetics of the coefficients: FP64, or double-float pairs.
// kBlocks: of an SM (double-float waits for its coefficients more than for a
// pipe: 38 x 46 x 36 with 198 directions 732 us with four, 684 with five, more
// with six, which spill; FP64 is bound by its pipe, 65^3 solve 430.9 ms with
// four, 432.0 with five).
struct AsmF64 {
    using V = double;
    static constexpr int kBlocks = 4;
    static __device__ __forceinline__ V zero() { return 0.0; }
    static __device__ __forceinline__ V weight(double w) { return w; }
    static __device__ __forceinline__ V fma(V w, V c, V a) { return ::fma(w, c, a); }
    static __device__ __forceinline__ V entry(V a) { return a; }
};
struct AsmDF {
    using V = float2;
    static constexpr int kBlocks = 5;
    static __device__ __forceinline__ V zero() { return make_float2(0.f, 0.f); }
    static __device__ __forceinline__ V weight(double w)
    {
        const dfl q = df_from_double(w);
        return make_float2(q.h, q.l);
    }
    // the sum is left unnormalised between contributions
    static __device__ __forceinline__ V fma(V w, V c, V a)
    {
        const dfl p = two_prod(w.x, c.x);
        const dfl s = two_sum(a.x, p.h);
        return make_float2(s.h, (a.y + s.l) + fmaf(w.y, c.x, fmaf(w.x, c.y, p.l)));
    }
    static __device__ __forceinline__ V entry(V a)
    {
        const dfl p = quick_two_sum(a.x, a.y);
        return make_float2(p.h, p.l);
    }
};

template <typename T>
__global__ void __launch_bounds__(kListThreads, T::kBlocks)
k_op_assemble(Geometry g, int r0, OpLists L, RecOut ro, const int* __restrict__ lmax, int nwp,
              const int* __restrict__ cnt, const int* __restrict__ segb, const int* __restrict__ E,
              const long long* __restrict__ eb, typename T::V* __restrict__ A)
{
    using V = typename T::V;
    // a contribution as every lane reads it: weight, row (kNoRow: none), element
    // of the entry that it completes (kOpen: none)
    struct __align__(16) Step {
        V wb;
        unsigned row, out;
    };
    constexpr unsigned kNoRow = ~0u, kOpen = ~0u;
    __shared__ Step steps[kListThreads / 32][32];
    extern __shared__ int2 lr[];     // [ndir] {length, first row}
    const int nz = g.nz, nxy = g.nx * g.ny;
    const int k0 = plane_at(g, r0 + blockIdx.y), tile = blockIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int t = tile * 32 + lane;
    const bool live = t < nxy;
    for (int d = threadIdx.x; d < g.ndir; d += blockDim.x)
        lr[d] = make_int2(lmax[((long long)d * nz + k0) * nwp + tile],
                          ro.rowbase[(long long)k0 * g.ndir + d]);
    __syncthreads();
    const char* c = reinterpret_cast<const char*>(reinterpret_cast<const V*>(ro.base) + ro.prow[k0] * nxy +
                                                  (live ? t : 0));
    const unsigned row_bytes = (unsigned)(nxy * sizeof(V));
    V* out = A + eb[k0] * (long long)nwp * 32 + (long long)tile * E[k0] * 32 + 2 * lane;
    Step* mine = steps[wid];
    int run = wid;                   // runs go round the warps, across the lists
    for (int q = blockIdx.z; q < 2 * nz; q += gridDim.z) {
        const int n = cnt[(long long)k0 * 2 * nz + q];
        if (n == 0) continue;
        const int m = q < nz ? q : q - nz;
        V* oq = out + (long long)segb[(long long)k0 * 2 * nz + q] * 32;
        const int* us = L.ustart + (long long)q * (L.ucap + 1);
        const OpContrib* ct = L.contrib + (long long)q * L.icap;
        const int runs = (n + kAsmRun - 1) / kAsmRun;
        for (; run < runs; run += nw) {
            const int js = us[run * kAsmRun], je = us[min(n, (run + 1) * kAsmRun)];
            V acc = T::zero();
            for (int jb = js; jb < je; jb += 32) {
                Step p{T::zero(), kNoRow, kOpen};
                if (jb + lane < je) {
                    const OpContrib k = ct[jb + lane];
                    const int2 r = lr[k.d];
                    if (m <= r.x || m == 0) p.row = r.y + m - 1 + ro.para;
                    p.wb = T::weight(k.wb);
                    // entry k.ul >> 1, in pairs of 32 x 2 elements
                    if (k.ul & 1) p.out = (unsigned)(k.ul >> 2) * 64 + ((k.ul >> 1) & 1);
                }
                __syncwarp();
                mine[lane] = p;
                __syncwarp();
                const int nj = min(32, je - jb);
                for (int i = 0; i < nj; i += 8) {
                    V cv[8];
#pragma unroll
                    for (int h = 0; h < 8; ++h) {
                        const unsigned r = mine[i + h].row;
                        cv[h] = T::zero();
                        if (live && r != kNoRow)
                            cv[h] = __ldg(reinterpret_cast<const V*>(c + (unsigned long long)r * row_bytes));
                    }
#pragma unroll
                    for (int h = 0; h < 8; ++h) {
                        const Step x = mine[i + h];
                        acc = T::fma(x.wb, cv[h], acc);
                        if (x.out != kOpen) {
                            oq[x.out] = T::entry(acc);
                            acc = T::zero();
                        }
                    }
                }
            }
            if ((n & 1) && (run + 1) * kAsmRun >= n) oq[(long long)(n >> 1) * 64 + 1] = T::zero();
        }
        run -= runs;
    }
    if (blockIdx.z) return;
    const int qz = 2 * nz - 1;
    const int tail = (segb[(long long)k0 * 2 * nz + qz] + cnt[(long long)k0 * 2 * nz + qz] + 1) / 2;
    for (int p = tail + wid; p < E[k0] / 2; p += nw)
        out[(long long)p * 64] = out[(long long)p * 64 + 1] = T::zero();
}

// c0[v] = sum over slots of c0s; bc[v] and ts[v] (when given) likewise (slot
// order fixed)
__global__ void k_op_own(long long N, const double* __restrict__ c0s, const double* __restrict__ bcs,
                         const double* __restrict__ tss, double* __restrict__ c0,
                         double* __restrict__ bc, double* __restrict__ ts)
{
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N;
         v += (long long)gridDim.x * blockDim.x) {
        double a = 0.0, b = 0.0, c = 0.0;
        for (int q = 0; q < kSlots; ++q) {
            a += c0s[q * N + v];
            b += bcs[q * N + v];
            if (tss) c += tss[q * N + v];
        }
        c0[v] = a;
        bc[v] = b;
        if (tss) ts[v] = c;
    }
}

// s, in planes padded to 2ny x 2nx by periodic copies, at voxel v: an entry's
// node is then at one offset from every voxel of the plane.
template <typename V>
__device__ __forceinline__ void pad_store(const Geometry& g, long long v, V s, V* __restrict__ sp)
{
    const int nx = g.nx, ny = g.ny;
    const long long W = 2LL * nx, P = 4LL * nx * ny;
    const int i = (int)(v % nx), j = (int)((v / nx) % ny);
    V* p = sp + v / ((long long)nx * ny) * P + (long long)j * W + i;
    p[0] = s;
    p[nx] = s;
    p[(long long)ny * W] = s;
    p[(long long)ny * W + nx] = s;
}
__device__ __forceinline__ void op_value(double s, double& x) { x = s; }
__device__ __forceinline__ void op_value(double s, float2& x)
{
    const dfl q = df_from_double(s);
    x = make_float2(q.h, q.l);
}

// The source in the apply kernel's form (V: double, or double-float pairs).
// With eps the source is formed here and written to S, in place of a kernel
// before this one (a kernel of a small grid costs its launch, 3 us).
template <typename V>
__global__ void k_op_pack(Geometry g, double* __restrict__ S, const double* __restrict__ eps,
                          const double* __restrict__ B, const double* __restrict__ J, V* __restrict__ sp)
{
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < g.N;
         v += (long long)gridDim.x * blockDim.x) {
        double s;
        if (eps) {
            const double e = eps[v];
            s = fma(e, B[v], (1.0 - e) * J[v]);
            S[v] = s;
        } else {
            s = S[v];
        }
        V x;
        op_value(s, x);
        pad_store(g, v, x, sp);
    }
}

// The sums of the NW warps of each of a cluster's C blocks added to a, in
// fixed order, by warp 0 of its first block (true there).
template <int NW, int C>
__device__ __forceinline__ bool tile_sum(double (&red)[NW][32], double mine, double& a)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    red[wid][lane] = mine;
    if constexpr (C == 1) {
        __syncthreads();
        if (wid != 0) return false;
        for (int w = 0; w < NW; ++w) a += red[w][lane];
        return true;
    } else {
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();
        const bool first = cl.block_rank() == 0 && wid == 0;
        if (first)
            for (int b = 0; b < C; ++b) {
                const double* r = cl.map_shared_rank(&red[0][0], b);
                for (int w = 0; w < NW; ++w) a += r[w * 32 + lane];
            }
        cl.sync();      // the blocks stay until their sums are read
        return first;
    }
}

// J of a source: C blocks (a cluster) per 32 voxels of a plane, their warps
// taking four entries at a time in turn (they stream the coefficients, 8 bytes
// per FP64 FMA, in order), then the warps' sums and the voxel's own terms in
// fixed order.  Bound by the FP64 pipe, so by the SM with the most work: tiles are
// split over a cluster where an SM has few.
template <int NWB, int C>
__global__ void __launch_bounds__(NWB * 32, 24 / NWB)
k_op_apply64(Geometry g, const double* __restrict__ S, const double* __restrict__ sp, OpMap op,
             double* __restrict__ J, unsigned long long* __restrict__ steps)
{
    constexpr int NW = NWB * C;
    __shared__ double red[NWB][32];
    const int nx = g.nx, nxy = nx * g.ny;
    const int tile = blockIdx.x, k0 = plane_at(g, blockIdx.y);
    const int lane = threadIdx.x & 31, wid = blockIdx.z * NWB + (threadIdx.x >> 5);
    const int t = tile * 32 + lane, tc = t < nxy ? t : 0;
    const int j0 = tc / nx, i0 = tc - j0 * nx;
    const long long at = (long long)k0 * 4 * nxy + (long long)j0 * 2 * nx + i0;
    const double* s = sp + at;
    const int E = op.E[k0];
    const long long eb = op.eb[k0];
    const double2* A = reinterpret_cast<const double2*>(op.A + eb * op.nwp * 32) +
                       (long long)tile * (E / 2) * 32 + lane;
    const int4* off = reinterpret_cast<const int4*>(op.off + eb);
    double acc0 = 0.0, acc1 = 0.0;
    constexpr int kQ = 4;       // quads of entries in flight per warp
    const int nq = E / 4;
    int q = wid;
    for (; q + (kQ - 1) * NW < nq; q += kQ * NW) {
        int4 o[kQ];
        double2 a[kQ], b[kQ];
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            o[i] = __ldg(off + q + i * NW);
            a[i] = __ldcs(A + (long long)(q + i * NW) * 64);
            b[i] = __ldcs(A + (long long)(q + i * NW) * 64 + 32);
        }
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            RT_GUARD(g, at + min(min(o[i].x, o[i].y), min(o[i].z, o[i].w)), 4 * g.N, kSiteFs64) continue;
            RT_GUARD(g, at + max(max(o[i].x, o[i].y), max(o[i].z, o[i].w)), 4 * g.N, kSiteFs64) continue;
            acc0 = fma(a[i].x, __ldg(s + o[i].x), acc0);
            acc1 = fma(a[i].y, __ldg(s + o[i].y), acc1);
            acc0 = fma(b[i].x, __ldg(s + o[i].z), acc0);
            acc1 = fma(b[i].y, __ldg(s + o[i].w), acc1);
        }
    }
    for (; q < nq; q += NW) {
        const int4 o = __ldg(off + q);
        RT_GUARD(g, at + min(min(o.x, o.y), min(o.z, o.w)), 4 * g.N, kSiteFs64) break;
        RT_GUARD(g, at + max(max(o.x, o.y), max(o.z, o.w)), 4 * g.N, kSiteFs64) break;
        const double2 a = __ldcs(A + (long long)q * 64), b = __ldcs(A + (long long)q * 64 + 32);
        acc0 = fma(a.x, __ldg(s + o.x), acc0);
        acc1 = fma(a.y, __ldg(s + o.y), acc1);
        acc0 = fma(b.x, __ldg(s + o.z), acc0);
        acc1 = fma(b.y, __ldg(s + o.w), acc1);
    }
    const long long v = (long long)k0 * nxy + tc;
    double a = fma(op.c0[v], S[v], op.bc[v]);
    if (tile_sum<NWB, C>(red, acc0 + acc1, a) && t < nxy) J[v] = a;
    if (steps && tile == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) atomicAdd(steps, *op.steps);
}

// h + l += (ah + al) ((sh + sl) - (s0h + s0l)): the difference of the high
// parts exact (TwoSum), the product's leading term split exactly, the sum of
// the leading parts exact (TwoSum); everything below goes to l.  h and l are
// not renormalised: l stays a sum of terms below 2^-23 of those in h.
__device__ __forceinline__ void diff_add_df(float& h, float& l, float ah, float al, float2 s,
                                            float s0h, float s0l)
{
    const dfl d = two_sum(s.x, -s0h);
    const float dl = d.l + (s.y - s0l);
    dfl p = two_prod(ah, d.h);
    p.l = fmaf(ah, dl, fmaf(al, d.h, p.l));
    const dfl t = two_sum(h, p.h);
    h = t.h;
    l += t.l + p.l;
}

// J of a source in double-float, as k_op_apply64 with the recording's
// difference form: J = sum_e A_e (S_e - S_0) + bc + (wsum - ts) S_0.  22
// FP32 operations and 8 coefficient bytes per entry: bound by memory.
template <int NW>
__global__ void __launch_bounds__(NW * 32, 32 / NW)
k_op_apply_df(Geometry g, const double* __restrict__ S, const float2* __restrict__ sp, OpMap op,
              double wsum, double* __restrict__ J, unsigned long long* __restrict__ steps)
{
    __shared__ double red[NW][32];
    const int nx = g.nx, nxy = nx * g.ny;
    const int tile = blockIdx.x, k0 = plane_at(g, blockIdx.y);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int t = tile * 32 + lane, tc = t < nxy ? t : 0;
    const int j0 = tc / nx, i0 = tc - j0 * nx;
    const long long at = (long long)k0 * 4 * nxy + (long long)j0 * 2 * nx + i0;
    const float2* s = sp + at;
    const float2 s0 = s[0];
    const int E = op.E[k0];
    const long long eb = op.eb[k0];
    const float4* A = reinterpret_cast<const float4*>(op.A + eb * op.nwp * 32) +
                      (long long)tile * (E / 2) * 32 + lane;
    const int4* off = reinterpret_cast<const int4*>(op.off + eb);
    float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
    constexpr int kQ = 2;       // quads of entries in flight per warp
    const int nq = E / 4;
    auto quad = [&](int4 o, float4 a, float4 b) {
        RT_GUARD(g, at + min(min(o.x, o.y), min(o.z, o.w)), 4 * g.N, kSiteFsdf) return;
        RT_GUARD(g, at + max(max(o.x, o.y), max(o.z, o.w)), 4 * g.N, kSiteFsdf) return;
        const float2 p0 = __ldg(s + o.x), p1 = __ldg(s + o.y), p2 = __ldg(s + o.z), p3 = __ldg(s + o.w);
        diff_add_df(h0, l0, a.x, a.y, p0, s0.x, s0.y);
        diff_add_df(h1, l1, a.z, a.w, p1, s0.x, s0.y);
        diff_add_df(h0, l0, b.x, b.y, p2, s0.x, s0.y);
        diff_add_df(h1, l1, b.z, b.w, p3, s0.x, s0.y);
    };
    int q = wid;
    for (; q + (kQ - 1) * NW < nq; q += kQ * NW) {
        int4 o[kQ];
        float4 a[kQ], b[kQ];
#pragma unroll
        for (int i = 0; i < kQ; ++i) {
            o[i] = __ldg(off + q + i * NW);
            a[i] = __ldcs(A + (long long)(q + i * NW) * 64);
            b[i] = __ldcs(A + (long long)(q + i * NW) * 64 + 32);
        }
#pragma unroll
        for (int i = 0; i < kQ; ++i) quad(o[i], a[i], b[i]);
    }
    for (; q < nq; q += NW)
        quad(__ldg(off + q), __ldcs(A + (long long)q * 64), __ldcs(A + (long long)q * 64 + 32));
    const long long v = (long long)k0 * nxy + tc;
    double a = op.bc[v];
    if (tile_sum<NW, 1>(red, ((double)h0 + (double)l0) + ((double)h1 + (double)l1), a) && t < nxy)
        J[v] = fma(wsum - op.ts[v], S[v], a);
    if (steps && tile == 0 && blockIdx.y == 0 && threadIdx.x == 0) atomicAdd(steps, *op.steps);
}

// Lambda* from the operator: the voxel's own coefficient and those of the
// nearest nodes of the neighbouring planes (distance 1 upstream; for the
// parabolic source also the downstream point).
template <bool DF>
__global__ void k_op_lstar(Geometry g, OpLists L, OpMap op, const int* __restrict__ cnt,
                           const int* __restrict__ segb, double* __restrict__ lstar)
{
    const int nxy = g.nx * g.ny, nz = g.nz;
    const int t = blockIdx.x * blockDim.x + threadIdx.x, k0 = blockIdx.y, o = blockIdx.z;
    if (t >= nxy) return;
    const long long v = (long long)k0 * nxy + t;
    const int oz = o / 9 - 1;
    double r = 0.0;
    if (oz == 0) {
        if (o == 13) r = op.c0[v];
    } else {
        const double* A = op.A + op.eb[k0] * (long long)op.nwp * 32 +
                          (long long)(t >> 5) * op.E[k0] * 32;
        for (int m = 1; m >= 0; --m) {
            // upstream (m = 1): plane k0 - s; downstream (m = 0): plane k0 + s
            const int si = (m == 1) == (oz < 0) ? 0 : 1;
            const int u = L.lpos[(si * 2 + m) * 9 + o % 9];
            const long long q = (long long)k0 * 2 * nz + (long long)si * nz + m;
            if (u < 0 || u >= cnt[q]) continue;
            const int e = segb[q] + u;
            const double* a = A + ((long long)(e >> 1) * 32 + (t & 31)) * 2 + (e & 1);
            if (DF) {
                const float2 p = *reinterpret_cast<const float2*>(a);
                r += (double)p.x + (double)p.y;
            } else {
                r += *a;
            }
        }
    }
    lstar[(long long)o * g.N + v] = r;
}

unsigned op_grid1d(long long n, int threads)
{
    long long b = (n + threads - 1) / threads;
    if (b > 152LL * 32) b = 152LL * 32;
    if (b < 1) b = 1;
    return (unsigned)b;
}

}  // namespace

// Nodes of a plane that fit in shared memory while its list is built.
constexpr int kListSmemNodes = 24 * 1024;

long long op_list_scratch(const Geometry& g)
{
    const long long nxy = (long long)g.nx * g.ny;
    return nxy <= kListSmemNodes ? 0 : 2 * nxy * g.nz;
}

cudaError_t launch_op_lists(const Geometry& g, const DirInfo* info, const StepGeo* off,
                            const Bw4d* bw, const DownGeo* dn, const OpLists& L, int* scratch,
                            cudaStream_t st)
{
    const size_t shm = scratch ? 0 : sizeof(int) * (size_t)g.nx * g.ny;
    if (shm > 40 * 1024) {
        // one value for all planes: contexts of several threads set it
        cudaError_t e = cudaFuncSetAttribute(k_op_lists, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(int) * kListSmemNodes);
        if (e != cudaSuccess) return e;
    }
    k_op_lists<<<2 * g.nz, kListThreads, shm, st>>>(g, info, off, bw, dn, L, scratch);
    return cudaGetLastError();
}

cudaError_t launch_op_lengths(const Geometry& g, const double* chi, const double* S,
                              const double* smax, const DirInfo* info, const int* poff,
                              const float4* bw32, double cut, int extra_bits, bool own, int groups,
                              float2* node, int* lmax, int nwp, int* Lp, unsigned long long* steps,
                              cudaStream_t st)
{
    if (own)
        k_op_pack_len<true><<<op_grid1d(g.N, 256), 256, 0, st>>>(g, chi, S, smax, node);
    else
        k_op_pack_len<false><<<op_grid1d(g.N, 256), 256, 0, st>>>(g, chi, S, smax, node);
    // two bits beyond the cutoff cover the FP32 rounding of tau and I
    const float lcut = cut > 0.0 ? (float)(-log2(cut)) + 2.0f + (float)extra_bits : INFINITY;
    // The directions are shared by more blocks than the march's (a ray here is
    // short, and the last wave of long blocks half empty): twice its groups, and
    // more until every SM has 32 blocks.  17^3 with 256 directions (FP64): solve 2.81
    // -> 2.76 ms; 33^3: first formal solution 4.09 -> 4.03; 38 x 46 x 36 with 198 (double-float) 2.26 ->
    // 2.22; half the march's groups 4.13 and 2.27; four times as the rule's.
    const int blocks = (g.nx * g.ny + kOpThreads - 1) / kOpThreads;
    int share = 2 * groups;
    while (share < g.ndir && (long long)blocks * g.nz * share < 152 * 32) share *= 2;
    const dim3 grid(blocks, share, g.nz);
    if (own)
        k_op_len<true><<<grid, kOpThreads, 0, st>>>(g, node, S, smax, info, poff, bw32, lcut, lmax, nwp);
    else
        k_op_len<false><<<grid, kOpThreads, 0, st>>>(g, node, S, smax, info, poff, bw32, lcut, lmax, nwp);
    cudaError_t e = cudaMemsetAsync(steps, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    k_op_plane_len<<<dim3((g.ndir + 7) / 8, g.nz), 256, 0, st>>>(g, lmax, nwp, Lp, steps);
    return cudaGetLastError();
}

cudaError_t launch_op_counts(const Geometry& g, const OpLists& L, bool para, const int* Lp,
                             int* rowbase, int* cnt, int* segb, int* E, int* rows, cudaStream_t st)
{
    k_op_counts<<<g.nz, kListThreads, 0, st>>>(g, L, para ? 1 : 0, Lp, rowbase, cnt, segb, E, rows);
    return cudaGetLastError();
}

cudaError_t launch_op_offsets(const Geometry& g, const OpLists& L, const int* cnt, const int* segb,
                              const OpMap& op, cudaStream_t st)
{
    const dim3 grid(2 * g.nz + 1 < 64 ? 2 * g.nz + 1 : 64, g.nz);
    k_op_offsets<<<grid, 128, 0, st>>>(g, L, cnt, segb, op.E, op.eb, const_cast<int*>(op.off));
    return cudaGetLastError();
}

cudaError_t launch_rec64(const Geometry& g, int r0, int nplanes, const double* chi, const double* B,
                         const double* G, const DirInfo* info, const StepGeo* off, const Bw4d* bw,
                         const Bw4d* bwh, const RecOut& ro, const int* lmax, int nwp, int groups,
                         double* c0s, double* bcs, cudaStream_t st)
{
    const dim3 grid((g.nx * g.ny + kOpThreads - 1) / kOpThreads, groups, nplanes);
    k_rec64<<<grid, kOpThreads, 0, st>>>(g, r0, chi, B, G, info, off, bw, bwh, ro, lmax, nwp, c0s,
                                         bcs);
    return cudaGetLastError();
}

cudaError_t launch_op_assemble(const Geometry& g, bool df, int r0, int nplanes, const OpLists& L,
                               const RecOut& ro, const int* lmax, const int* cnt, const int* segb,
                               const OpMap& op, cudaStream_t st)
{
    const size_t shm = sizeof(int2) * (size_t)g.ndir;
    if (shm > 48 * 1024) {
        // one value for all quadratures: contexts of several threads set it
        cudaError_t e = df ? cudaFuncSetAttribute(k_op_assemble<AsmDF>,
                                                  cudaFuncAttributeMaxDynamicSharedMemorySize, kAsmShared)
                           : cudaFuncSetAttribute(k_op_assemble<AsmF64>,
                                                  cudaFuncAttributeMaxDynamicSharedMemorySize, kAsmShared);
        if (e != cudaSuccess) return e;
    }
    // few tiles: several blocks share a tile's lists, so that every SM has
    // work (17^3 with 256 directions: 93 against 258 us)
    int split = 1;
    while (split < 8 && (long long)op.nwp * nplanes * split < 152 * 8) split *= 2;
    const dim3 grid(op.nwp, nplanes, split);
    double* A = const_cast<double*>(op.A);
    if (df)
        k_op_assemble<AsmDF><<<grid, kListThreads, shm, st>>>(g, r0, L, ro, lmax, op.nwp, cnt, segb, op.E,
                                                              op.eb, reinterpret_cast<float2*>(A));
    else
        k_op_assemble<AsmF64><<<grid, kListThreads, shm, st>>>(g, r0, L, ro, lmax, op.nwp, cnt, segb,
                                                               op.E, op.eb, A);
    return cudaGetLastError();
}

cudaError_t launch_op_own(long long N, const double* c0s, const double* bcs, const double* tss,
                          const OpMap& op, cudaStream_t st)
{
    k_op_own<<<op_grid1d(N, 256), 256, 0, st>>>(N, c0s, bcs, tss, const_cast<double*>(op.c0),
                                                const_cast<double*>(op.bc), const_cast<double*>(op.ts));
    return cudaGetLastError();
}

namespace {
// The tiles of the grid with clusters of C blocks per tile.
template <int NWB, int C, typename K, typename... P>
cudaError_t launch_tiles(K kernel, dim3 tiles, cudaStream_t st, P... p)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(tiles.x, tiles.y, C);
    cfg.blockDim = dim3(NWB * 32);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = at.val.clusterDim.y = 1;
    at.val.clusterDim.z = C;
    cfg.attrs = &at;
    cfg.numAttrs = C > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, p...);
}
}  // namespace

// How many warps share a tile.  FP64 (the SM with the most work ends it):
// formal solution of 33^3 with 256 directions (1155 tiles) 367 us with one block
// of eight warps per tile, 343 with two; 48^3 (3456) 1.38 against 1.37 ms, but
// 65^3 (8645) 4.58 against 4.61; 17^3 (170) like one block of 16 warps.
// Double-float (memory, one block): 33^3 319 us with eight warps, 269 with 16;
// 41^3 616 / 555; 48^3 and 65^3 the same.
constexpr long long kManyTiles = 4096;

cudaError_t launch_op_pack(const Geometry& g, double* S, const double* eps, const double* B,
                           const double* J, bool df, double* sp, cudaStream_t st)
{
    const unsigned n = op_grid1d(g.N, 256);
    if (df)
        k_op_pack<<<n, 256, 0, st>>>(g, S, eps, B, J, reinterpret_cast<float2*>(sp));
    else
        k_op_pack<<<n, 256, 0, st>>>(g, S, eps, B, J, sp);
    return cudaGetLastError();
}

cudaError_t launch_op_apply64(const Geometry& g, const double* S, const double* sp, const OpMap& op,
                              double* J, unsigned long long* steps, cudaStream_t st)
{
    const dim3 tiles(op.nwp, g.nz);
    if ((long long)op.nwp * g.nz < kManyTiles)
        return launch_tiles<8, 2>(k_op_apply64<8, 2>, tiles, st, g, S, sp, op, J, steps);
    return launch_tiles<8, 1>(k_op_apply64<8, 1>, tiles, st, g, S, sp, op, J, steps);
}

cudaError_t launch_op_apply_df(const Geometry& g, const double* S, const double* sp, const OpMap& op,
                               double wsum, double* J, unsigned long long* steps, cudaStream_t st)
{
    const float2* p = reinterpret_cast<const float2*>(sp);
    const dim3 tiles(op.nwp, g.nz);
    if ((long long)op.nwp * g.nz < kManyTiles)
        return launch_tiles<16, 1>(k_op_apply_df<16>, tiles, st, g, S, p, op, wsum, J, steps);
    return launch_tiles<8, 1>(k_op_apply_df<8>, tiles, st, g, S, p, op, wsum, J, steps);
}

cudaError_t launch_op_lstar(const Geometry& g, bool df, const OpLists& L, const OpMap& op,
                            const int* cnt, const int* segb, double* lstar, cudaStream_t st)
{
    const dim3 grid((g.nx * g.ny + 127) / 128, g.nz, 27);
    if (df)
        k_op_lstar<true><<<grid, 128, 0, st>>>(g, L, op, cnt, segb, lstar);
    else
        k_op_lstar<false><<<grid, 128, 0, st>>>(g, L, op, cnt, segb, lstar);
    return cudaGetLastError();
}

}  // namespace rt3d
