// Short characteristics with recorded weights (see sc.cu for the method:
// Hauschildt & Baron 2011, Sect. 2.2, O(1) per voxel and direction).
//
// The weights of every (voxel, direction) depend on the opacities only, so
// they are computed once per opacity, with no order between the planes
// ([direction][plane][voxel]); a formal solution then walks the planes of
// each direction with two bilinear interpolations and a few operations per
// node instead of three interpolations, an exponential and a division.
//   FP64 (24 bytes: w_cur, e and w_up): I = e I(p) + w_cur S + w_up S(p),
//     J = sum_d w_d I_d;
//   double-float (a value a pair of floats; 16 bytes: w_cur and e): the
//     deviation D = I - S from the source at the node as in the
//     double-float march, D = e D(p) + (1 - w_cur) (S(p) - S), w_up + e being
//     1 - w_cur, J = (sum_d w_d) S + sum_d w_d D_d.
// The sums over the directions run in direction order.
//
// Mapping as in sc.cu: one block per direction, the preceding and the current
// plane of D in shared memory (or in a global scratch), a barrier per plane;
// each block writes I (D) to its slice of a [directions][N] buffer.
#include "dfweights.cuh"
#include "internal.h"
#include "weights.cuh"

namespace rt3d {

namespace {

constexpr int kRecThreads = 128;

struct ScCorners {
    int a00, a10, a01, a11;
};

__device__ __forceinline__ ScCorners sc_corners(int i, int j, StepGeo o, int nx, int ny)
{
    int x0 = i + o.ox;
    x0 -= x0 >= nx ? nx : 0;
    const int x1 = x0 + 1 == nx ? 0 : x0 + 1;
    int y0 = j + o.oy;
    y0 -= y0 >= ny ? ny : 0;
    const int y1 = y0 + 1 == ny ? 0 : y0 + 1;
    return ScCorners{y0 * nx + x0, y0 * nx + x1, y1 * nx + x0, y1 * nx + x1};
}

__device__ __forceinline__ bool sc_inside(const Geometry& g, ScCorners c, int site)
{
    RT_GUARD(g, max(max(c.a00, c.a10), max(c.a01, c.a11)), g.nx * g.ny, site) return false;
    RT_GUARD(g, min(min(c.a00, c.a10), min(c.a01, c.a11)), g.nx * g.ny, site) return false;
    return true;
}

struct Sc64 {
    using V = double;
    using C = double2;      // {w_cur, e}; w_up follows in an array of its own
    struct Coef {
        double2 a;
        double u;
    };
    using W = Bw4d;
    static constexpr bool kDiff = false;
    // threads of a block of the apply kernel, nodes in flight per thread:
    // bound by the FP64 pipe, 65^3 x 1024 formal solution 6.16 ms with 384
    // threads and one node (6.43 with 256, 6.76 with two nodes)
    static constexpr int kThreads = 384, kUnroll = 1;
    static constexpr int kTab = kExpTable;
    using T = double;
    static __device__ __forceinline__ void fill(T* t) { fill_exp_table(t); }
    static __device__ __forceinline__ W weights(const ScView& p, int d) { return p.bw[(long long)d * p.g.nz + 1]; }
    static __device__ __forceinline__ V zero() { return 0.0; }
    static __device__ __forceinline__ V make(double x) { return x; }
    static __device__ __forceinline__ double value(V x) { return x; }
    static __device__ __forceinline__ V bilin(W b, V a, V c, V d, V e) { return b.x * a + b.y * c + b.z * d + b.w * e; }
    // optical depth of the segment between nodes of opacity a and c
    static __device__ __forceinline__ V depth(const DirInfo& di, V a, V c) { return di.hs * (a + c); }
    static __device__ __forceinline__ void segment(V x, const T* tab, V& wc, V& wu, V& e) { seg_weights64(x, tab, wc, wu, e); }
    static __device__ __forceinline__ void store(C* c, long long n, long long i, V wc, V wu, V e)
    {
        __stcs(c + i, make_double2(wc, e));
        __stcs(reinterpret_cast<double*>(c + n) + i, wu);
    }
    static __device__ __forceinline__ Coef load(const C* c, long long n, long long i)
    {
        return Coef{__ldcs(c + i), __ldcs(reinterpret_cast<const double*>(c + n) + i)};
    }
    static __device__ __forceinline__ V wcur(C c) { return c.x; }
    static __device__ __forceinline__ V step(Coef c, V Ip, V Sp, V S)
    {
        return fma(c.a.y, Ip, fma(c.a.x, S, c.u * Sp));
    }
    static __device__ __forceinline__ V mul(V a, V b) { return a * b; }
    static __device__ __forceinline__ V add(V a, V b) { return a + b; }
    // the direction sum of eight
    struct Acc {
        double s;
    };
    static __device__ __forceinline__ void acc(Acc& a, V w, V D) { a.s = fma(w, D, a.s); }
    static __device__ __forceinline__ double sum(Acc a) { return a.s; }
};

struct ScDF {
    using V = float2;
    using C = float4;       // {w_cur, e}, each a pair
    using Coef = float4;
    static constexpr bool kDiff = true;
    // bound by the latency between the barriers of the planes: 65^3 x 1024
    // formal solution 3.26 ms with 256 threads, 2.75 with 384, 2.51 with 512,
    // 2.39 with 640, 3.3 with 768 (whose registers leave one block per SM)
    static constexpr int kThreads = 640, kUnroll = 2;
    struct W {
        float4 h, l;
    };
    static constexpr int kTab = 2 * kExpTableDF;
    using T = dfl;
    static __device__ __forceinline__ dfl d(V v) { return df_make(v.x, v.y); }
    static __device__ __forceinline__ V v(dfl x) { return make_float2(x.h, x.l); }
    static __device__ __forceinline__ void fill(T* t) { fill_exp_table_df(t); }
    static __device__ __forceinline__ W weights(const ScView& p, int dir)
    {
        const float4* q = p.bwdf + 2 * ((long long)dir * p.g.nz + 1);
        return W{q[0], q[1]};
    }
    static __device__ __forceinline__ V zero() { return make_float2(0.f, 0.f); }
    static __device__ __forceinline__ V make(double x) { return v(df_from_double(x)); }
    static __device__ __forceinline__ double value(V x) { return (double)x.x + (double)x.y; }
    static __device__ __forceinline__ V bilin(W w, V a, V b, V c, V e)
    {
        return v(bilin_df(w.h, w.l, a.x, a.y, b.x, b.y, c.x, c.y, e.x, e.y));
    }
    static __device__ __forceinline__ V depth(const DirInfo& di, V a, V c)
    {
        return v(df_mul(df_make(di.hs32, di.hs32lo), df_add_s(d(a), d(c))));
    }
    static __device__ __forceinline__ void segment(V x, const T* tab, V& wc, V& wu, V& e)
    {
        dfl a, b, c;
        seg_weights_df(d(x), tab, a, b, c);
        wc = v(a);
        wu = v(b);
        e = v(c);
    }
    static __device__ __forceinline__ void store(C* c, long long, long long i, V wc, V, V e)
    {
        __stcs(c + i, make_float4(wc.x, wc.y, e.x, e.y));
    }
    static __device__ __forceinline__ Coef load(const C* c, long long, long long i) { return __ldcs(c + i); }
    static __device__ __forceinline__ V wcur(C c) { return make_float2(c.x, c.y); }
    static __device__ __forceinline__ V step(Coef c, V Dp, V Sp, V S)
    {
        const dfl q = df_sub_s(d(Sp), d(S));
        const dfl k = df_add_f(df_make(-c.x, -c.y), 1.0f);
        return v(df_add_s(df_mul(df_make(c.z, c.w), d(Dp)), df_mul(k, q)));
    }
    static __device__ __forceinline__ V mul(V a, V b) { return v(df_mul(d(a), d(b))); }
    static __device__ __forceinline__ V add(V a, V b) { return v(df_add_s(d(a), d(b))); }
    struct Acc {
        float h, l;
    };
    static __device__ __forceinline__ void acc(Acc& a, V w, V D)
    {
        const dfl p = two_prod(w.x, D.x);
        const dfl s = two_sum(a.h, p.h);
        a.h = s.h;
        a.l += s.l + fmaf(w.y, D.x, fmaf(w.x, D.y, p.l));
    }
    static __device__ __forceinline__ double sum(Acc a) { return (double)a.h + (double)a.l; }
};

// chi in the form's arithmetic (double-float: unpadded pairs, else chi itself)
template <typename A>
__device__ __forceinline__ const typename A::V* sc_chi(const ScView& p);
template <>
__device__ __forceinline__ const double* sc_chi<Sc64>(const ScView& p)
{
    return p.chi;
}
template <>
__device__ __forceinline__ const float2* sc_chi<ScDF>(const ScView& p)
{
    return p.chi2;
}
template <typename A>
__device__ __forceinline__ const typename A::V* sc_src(const ScView& p);
template <>
__device__ __forceinline__ const double* sc_src<Sc64>(const ScView& p)
{
    return p.S;
}
template <>
__device__ __forceinline__ const float2* sc_src<ScDF>(const ScView& p)
{
    return p.S2;
}

// Bilinear weight of corner q.
__device__ __forceinline__ double sc_corner_weight(const Bw4d& b, int q)
{
    return q == 0 ? b.x : q == 1 ? b.y : q == 2 ? b.z : b.w;
}
__device__ __forceinline__ float2 sc_corner_weight(const ScDF::W& b, int q)
{
    return q == 0 ? make_float2(b.h.x, b.l.x) : q == 1 ? make_float2(b.h.y, b.l.y)
         : q == 2 ? make_float2(b.h.z, b.l.z) : make_float2(b.h.w, b.l.w);
}

// x as double-float pairs
__global__ void k_sc_pairs(long long N, const double* __restrict__ x, float2* __restrict__ out)
{
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N;
         v += (long long)gridDim.x * blockDim.x) {
        const dfl q = df_from_double(x[v]);
        out[v] = make_float2(q.h, q.l);
    }
}

// w_cur and e of every (direction, voxel) off the entry plane.
template <typename A>
__global__ void __launch_bounds__(kRecThreads)
k_sc_rec(ScView p, typename A::C* __restrict__ coef)
{
    __shared__ typename A::T tab[A::kTab];
    A::fill(tab);
    __syncthreads();
    const Geometry& g = p.g;
    const int nxy = g.nx * g.ny, nz = g.nz;
    const int t = blockIdx.x * kRecThreads + threadIdx.x, k = blockIdx.y;
    if (t >= nxy) return;
    const int j = t / g.nx, i = t - j * g.nx;
    const typename A::V* chi = sc_chi<A>(p);
    const typename A::V me = chi[(long long)k * nxy + t];
    for (int d = blockIdx.z; d < g.ndir; d += gridDim.z) {
        const DirInfo di = p.info[d];
        const int ku = k - di.sgn;
        if (ku < 0 || ku >= nz) continue;
        const ScCorners c = sc_corners(i, j, p.off[(long long)d * nz + 1], g.nx, g.ny);
        if (!sc_inside(g, c, kSiteSc)) continue;
        const typename A::V* u = chi + (long long)ku * nxy;
        const auto b = A::weights(p, d);
        const auto cu = A::bilin(b, __ldg(u + c.a00), __ldg(u + c.a10), __ldg(u + c.a01), __ldg(u + c.a11));
        typename A::V wc, wu, e;
        A::segment(A::depth(di, cu, me), tab, wc, wu, e);
        A::store(coef, g.ndir * g.N, ((long long)d * nz + k) * nxy + t, wc, wu, e);
    }
}

template <typename A, bool SMEM, int kScrThreads>
__global__ void __launch_bounds__(kScrThreads)
k_sc_apply(ScView p, const typename A::C* __restrict__ coef, int d0, typename A::V* __restrict__ part,
           typename A::V* gplanes, unsigned long long* __restrict__ steps)
{
    using V = typename A::V;
    extern __shared__ double2 splanes_raw[];
    const Geometry& g = p.g;
    const int nx = g.nx, ny = g.ny, nz = g.nz, nxy = nx * ny;
    const int d = d0 + blockIdx.x;
    V* pl = SMEM ? reinterpret_cast<V*>(splanes_raw) : gplanes + (long long)blockIdx.x * 2 * nxy;
    const DirInfo di = p.info[d];
    const int s = di.sgn;
    const StepGeo o = p.off[(long long)d * nz + 1];
    const auto b = A::weights(p, d);
    const int bc = s > 0 ? g.top_bc : g.bottom_bc, kin = s > 0 ? 0 : nz - 1;
    V* out = part + (long long)blockIdx.x * g.N;
    const V* src = sc_src<A>(p);
    for (int t = threadIdx.x; t < nxy; t += kScrThreads) {
        double I = 0.0;
        if (bc) {
            I = p.B[(long long)kin * nxy + t];
            if (bc == 2) I = fma(di.amu, p.G[t], I);
        }
        const V D = A::make(A::kDiff ? I - p.S[(long long)kin * nxy + t] : I);
        pl[t] = D;
        out[(long long)kin * nxy + t] = D;
    }
    __syncthreads();
    const int dj = kScrThreads / nx, di0 = kScrThreads - dj * nx;
    const int jf = threadIdx.x / nx, if0 = threadIdx.x - jf * nx;
    int cur = 0;
    for (int n = 1; n < nz; ++n) {
        const int k = s > 0 ? n : nz - 1 - n;
        const V* prev = pl + cur * nxy;
        V* next = pl + (cur ^ 1) * nxy;
        const V* Sk = src + (long long)k * nxy;
        const V* Su = src + (long long)(k - s) * nxy;
        const long long ck = ((long long)d * nz + k) * nxy;
        V* outk = out + (long long)k * nxy;
        int i = if0, j = jf;
#pragma unroll (A::kUnroll)
        for (int t = threadIdx.x; t < nxy; t += kScrThreads) {
            const ScCorners c = sc_corners(i, j, o, nx, ny);
            i += di0;
            j += dj;
            if (i >= nx) {
                i -= nx;
                ++j;
            }
            if (!sc_inside(g, c, kSiteSc)) continue;
            const auto cf = A::load(coef, g.ndir * g.N, ck + t);
            const V Sp = A::bilin(b, __ldg(Su + c.a00), __ldg(Su + c.a10), __ldg(Su + c.a01),
                                  __ldg(Su + c.a11));
            const V Dp = A::bilin(b, prev[c.a00], prev[c.a10], prev[c.a01], prev[c.a11]);
            const V D = A::step(cf, Dp, Sp, __ldg(Sk + t));
            next[t] = D;
            outk[t] = D;
        }
        __syncthreads();
        cur ^= 1;
    }
    if (steps && threadIdx.x == 0) atomicAdd(steps, (unsigned long long)(nz - 1) * nxy);
}

// J[v] = (accumulate ? J[v] : wsum S[v], or 0 when the slices hold I) + sum
// over q < nd of w_{d0+q} part[q][v]; eight directions at a time in the form's
// arithmetic, their sums in FP64.
template <typename A>
__global__ void __launch_bounds__(256)
k_sc_sum(ScView p, int d0, int nd, const typename A::V* __restrict__ part, double wsum,
         double* __restrict__ J, int accumulate)
{
    extern __shared__ double2 sw_raw[];
    typename A::V* sw = reinterpret_cast<typename A::V*>(sw_raw);
    for (int q = threadIdx.x; q < nd; q += blockDim.x) sw[q] = A::make(p.info[d0 + q].w);
    __syncthreads();
    const long long N = p.g.N;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N;
         v += (long long)gridDim.x * blockDim.x) {
        double s = accumulate ? J[v] : A::kDiff ? wsum * p.S[v] : 0.0;
        int q = 0;
        for (; q + 8 <= nd; q += 8) {
            typename A::V x[8];
            typename A::Acc a{};
#pragma unroll
            for (int h = 0; h < 8; ++h) x[h] = __ldcs(part + (long long)(q + h) * N + v);
#pragma unroll
            for (int h = 0; h < 8; ++h) A::acc(a, sw[q + h], x[h]);
            s += A::sum(a);
        }
        for (; q < nd; ++q) {
            typename A::Acc a{};
            A::acc(a, sw[q], part[(long long)q * N + v]);
            s += A::sum(a);
        }
        J[v] = s;
    }
}

// Lambda* from the recorded weights (see k_lstar_sc64): per direction w_cur at
// the voxel and, at the corners c of its upstream point, b_c (w_up + e
// w_cur(c)), w_cur(c) read from c's own record (0 on the entry plane).  FP64
// reads the voxel's own weights as well (65^3 x 1024: 4.9 ms, 14.4 forming them
// again); double-float, whose record has no w_up, forms them.
template <typename A>
__global__ void __launch_bounds__(kRecThreads)
k_sc_lstar(ScView p, const typename A::C* __restrict__ coef, double* __restrict__ lstar)
{
    using V = typename A::V;
    __shared__ V lam[27][kRecThreads];
    __shared__ typename A::T tab[A::kDiff ? A::kTab : 1];
    for (int q = 0; q < 27; ++q) lam[q][threadIdx.x] = A::zero();
    if (A::kDiff) {
        A::fill(tab);
        __syncthreads();
    }
    const Geometry& g = p.g;
    const int nxy = g.nx * g.ny, nz = g.nz;
    const int t = blockIdx.x * kRecThreads + threadIdx.x, k = blockIdx.y;
    if (t >= nxy) return;
    const int j = t / g.nx, i = t - j * g.nx;
    const V* chi = sc_chi<A>(p);
    const V me = chi[(long long)k * nxy + t];
    for (int d = 0; d < g.ndir; ++d) {
        const DirInfo di = p.info[d];
        const int ku = k - di.sgn;
        if (ku < 0 || ku >= nz) continue;
        const ScCorners c = sc_corners(i, j, p.off[(long long)d * nz + 1], g.nx, g.ny);
        if (!sc_inside(g, c, kSiteLstarSc)) continue;
        const auto b = A::weights(p, d);
        V wc, wu, e;
        if constexpr (A::kDiff) {
            const V* u = chi + (long long)ku * nxy;
            A::segment(A::depth(di, A::bilin(b, __ldg(u + c.a00), __ldg(u + c.a10), __ldg(u + c.a01),
                                             __ldg(u + c.a11)), me), tab, wc, wu, e);
        } else {
            const auto own = A::load(coef, g.ndir * g.N, ((long long)d * nz + k) * nxy + t);
            wc = own.a.x;
            e = own.a.y;
            wu = own.u;
        }
        const V wd = A::make(di.w);
        lam[13][threadIdx.x] = A::add(lam[13][threadIdx.x], A::mul(wd, wc));
        const bool deeper = ku != (di.sgn > 0 ? 0 : nz - 1);
        const typename A::C* cu = coef + ((long long)d * nz + ku) * nxy;
        const int cn[4] = {c.a00, c.a10, c.a01, c.a11};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int lo = di.lo[q];
            if (lo < 0) continue;
            V x = wu;
            if (deeper) x = A::add(wu, A::mul(e, A::wcur(__ldg(cu + cn[q]))));
            lam[lo][threadIdx.x] = A::add(lam[lo][threadIdx.x], A::mul(A::mul(wd, sc_corner_weight(b, q)), x));
        }
    }
    for (int q = 0; q < 27; ++q) lstar[(long long)q * g.N + (long long)k * nxy + t] = A::value(lam[q][threadIdx.x]);
}

template <typename A>
cudaError_t sc_record(const ScView& p, void* coef, cudaStream_t st)
{
    const int tiles = (p.g.nx * p.g.ny + kRecThreads - 1) / kRecThreads;
    int G = 1;      // blocks that share a tile's directions: enough to fill the GPU
    while (G < 64 && 2 * G <= p.g.ndir && (long long)tiles * p.g.nz * G < 152 * 64) G *= 2;
    k_sc_rec<A><<<dim3(tiles, p.g.nz, G), kRecThreads, 0, st>>>(p, static_cast<typename A::C*>(coef));
    return cudaGetLastError();
}

// T threads: not more warps than a plane has work for, so that more directions share
// an SM (formal solution of 9 x 9 x 129 with 4096 directions 2.36 ms with 640 threads, 1.36
// with 128 in double-float, 2.35 and 1.70 in FP64; the march without a recording takes
// 2.17 and 4.2).  A constant: with the number from blockDim 65^3 x 1024 took 7% longer.
template <typename A, bool SMEM, int T>
cudaError_t sc_apply(const ScView& p, const void* coef, double wsum, void* part, void* gplanes, double* J,
                     unsigned long long* steps, cudaStream_t st)
{
    const Geometry& g = p.g;
    const int chunk = sc_chunk(g);
    const size_t shm = SMEM ? 16 * (size_t)g.nx * g.ny : 0;
    if (shm > 40 * 1024) {
        // one value for all grids: contexts of several threads set it
        cudaError_t e = cudaFuncSetAttribute(k_sc_apply<A, SMEM, T>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
    }
    long long rb = (g.N + 255) / 256;
    if (rb > 152LL * 16) rb = 152LL * 16;
    auto* c = static_cast<const typename A::C*>(coef);
    auto* pt = static_cast<typename A::V*>(part);
    auto* gp = static_cast<typename A::V*>(gplanes);
    for (int d0 = 0; d0 < g.ndir; d0 += chunk) {
        const int nd = g.ndir - d0 < chunk ? g.ndir - d0 : chunk;
        k_sc_apply<A, SMEM, T><<<nd, T, shm, st>>>(p, c, d0, pt, gp, steps);
        k_sc_sum<A><<<(unsigned)rb, 256, sizeof(typename A::V) * nd, st>>>(p, d0, nd, pt, wsum, J, d0 > 0);
    }
    return cudaGetLastError();
}

template <typename A>
cudaError_t sc_apply_any(const ScView& p, const void* coef, double wsum, void* part, void* gplanes, double* J,
                         unsigned long long* steps, cudaStream_t st)
{
    const int nxy = p.g.nx * p.g.ny;
    if (sc_scratch_planes(p.g)) return sc_apply<A, false, A::kThreads>(p, coef, wsum, part, gplanes, J, steps, st);
    if (nxy <= 128) return sc_apply<A, true, 128>(p, coef, wsum, part, gplanes, J, steps, st);
    if (nxy <= 256) return sc_apply<A, true, 256>(p, coef, wsum, part, gplanes, J, steps, st);
    return sc_apply<A, true, A::kThreads>(p, coef, wsum, part, gplanes, J, steps, st);
}

}  // namespace

cudaError_t launch_sc_pairs(long long N, const double* x, float2* out, cudaStream_t st)
{
    long long b = (N + 255) / 256;
    if (b > 152LL * 32) b = 152LL * 32;
    k_sc_pairs<<<(unsigned)b, 256, 0, st>>>(N, x, out);
    return cudaGetLastError();
}

cudaError_t launch_sc_record(const ScView& p, bool df, void* coef, cudaStream_t st)
{
    return df ? sc_record<ScDF>(p, coef, st) : sc_record<Sc64>(p, coef, st);
}

cudaError_t launch_sc_apply(const ScView& p, bool df, const void* coef, double wsum, void* part,
                            void* gplanes, double* J, unsigned long long* steps, cudaStream_t st)
{
    return df ? sc_apply_any<ScDF>(p, coef, wsum, part, gplanes, J, steps, st)
              : sc_apply_any<Sc64>(p, coef, wsum, part, gplanes, J, steps, st);
}

cudaError_t launch_sc_lstar(const ScView& p, bool df, const void* coef, double* lstar, cudaStream_t st)
{
    const dim3 grid((p.g.nx * p.g.ny + kRecThreads - 1) / kRecThreads, p.g.nz);
    if (df)
        k_sc_lstar<ScDF><<<grid, kRecThreads, 0, st>>>(p, static_cast<const float4*>(coef), lstar);
    else
        k_sc_lstar<Sc64><<<grid, kRecThreads, 0, st>>>(p, static_cast<const double2*>(coef), lstar);
    return cudaGetLastError();
}

}  // namespace rt3d
