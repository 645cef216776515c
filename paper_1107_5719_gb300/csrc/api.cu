// C ABI of librt3d.so (declared in include/rt3d.h): the context, argument
// checks, device buffers and the host-side driver of the outer iteration
// (Hauschildt & Baron 2011, Sect. 2: formal solution -> operator splitting,
// everything resident on the GPU, only inputs and J cross the bus).
#include "../../include/rt3d.h"
#include "internal.h"

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <algorithm>
#include <vector>

using namespace rt3d;

struct rt_ctx {
    int device = 0;
    int precision = RT_FP64;
    cudaStream_t own_stream = nullptr;
    cudaStream_t stream = nullptr;
    int num_sms = 0;

    Geometry g{};
    double dx = 1, dy = 1, dz = 1;
    bool have_grid = false, have_quad = false, have_chi = false, have_eps = false, have_B = false;
    bool lstar_valid = false, coef_valid = false, b2_valid = false;
    int os_method = RT_OS_JACOBI;
    double df_switch = 0.0;   // FP32 sweep: finishing stage once delta < this
    // Finishing stage of an FP32-sweep solve: 0 off; 1 the next formal
    // solution is the double-float reference J_ref = J_FS(S_ref) of the
    // current source; 2 formal solutions march the source change
    // dS = S - S_ref in FP32 and add it: J_FS(S) = J_ref + J_FS(dS) with zero
    // boundary intensities (the formal solution is linear in S).
    int fin = 0;
    double *S_ref = nullptr, *J_ref = nullptr, *dS = nullptr;
    // operator-splitting step as a CUDA graph with the sweep loop in a WHILE
    // node (two cached instances: J_old alternates between two buffers)
    struct OsGraph {
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        const double* jold = nullptr;
        const double* jfs = nullptr;
        const double* jnew = nullptr;
        const double* dlt = nullptr;
        int max_sweeps = 0, method = -1;
        double tol = -1.0;
    } osg[2];
    int osg_next = 0;
    int* d_nsw = nullptr;     // the graph's sweep counter
    int* d_sw = nullptr;      // sweeps of the last OS step (behind scal), and a pinned copy
    int* h_sw = nullptr;
    bool os_one = false;      // the last step ran as one kernel (launch_os_solve)
    // its barrier words: two sets in turn, each zeroed by the solve before the
    // one that uses it; words in use and of each set not zero
    unsigned long long* os_words = nullptr;
    int os_cap = 0, os_set = 0, os_dirty[2] = {0, 0};
    // where that kernel forms the outer delta and copies J_old to, in a solve's
    // iterations without extrapolation (null: it does not)
    double *os_delta = nullptr, *os_hist = nullptr;
    bool use_graphs = true;
    unsigned long long* berr = nullptr;   // checked builds: out-of-bounds record
    int fs_method = RT_FS_LONG;
    int src_order = RT_SRC_LINEAR;
    DownGeo* dn = nullptr;   // downstream-point table (FP64 contexts)
    double *scpart = nullptr, *scplanes = nullptr;   // short characteristics
    size_t scpart_n = 0, scplanes_n = 0;
    int groups_req = 0;
    int threads32 = 0;       // threads per block of the FP32 march (0: 128)
    int order32 = 0;         // block order of the FP32 march (0 auto, 1 tile-, 2 plane-major)
    double cut = -1.0;
    // recorded FP64 march (FsRec): the first formal solution after the
    // opacities, directions or boundary change records it, later ones
    // replay it.  rec_mode: -1 automatic, 0 off, > 0 a byte limit.
    long long rec_mode = -1;
    FsRec rec{};
    Rec32 rec32{};              // the FP32-sweep recording (same memory block)
    float2* srec = nullptr;    // the replay's source records
    char* rec_mem = nullptr;
    long long rec_cap = 0;
    bool rec_valid = false;
    // the recording assembled into an operator (rec_op), in the same block;
    // its node lists (per quadrature) and the recording's working storage
    bool rec_op = false;
    bool op_packed = false;     // the source of the coming formal solution is packed (operator, replay)
    bool op_steps = false;      // h_steps holds the recording's steps
    OpMap op{};
    OpLists ol{};
    // (blocks kept over a change of the quadrature; ok: made for this one)
    char *ol_mem = nullptr, *ow_mem = nullptr;
    long long ol_cap = 0, ow_cap = 0;
    bool ol_ok = false, ow_ok = false;
    int ow_bounds = -1;         // eb and prow on the device: op_bounds without (0) or with (1) para
    struct OpWork {
        double* sp;             // padded source planes (also the length march's nodes)
        int *lmax, *Lp, *rowbase, *cnt, *segb, *E, *rows, *poff;
        long long *eb, *prow;
        unsigned long long* steps;
        double *c0s, *bcs, *tss;
    } ow{};
    std::vector<int> dord;      // directions by sign and decreasing |mu| (OpLists)
    int dpos = 0;

    // device state, FP64
    double *chi = nullptr, *eps = nullptr, *B = nullptr, *J = nullptr, *S = nullptr;
    double *Jfs = nullptr, *Jn = nullptr, *Ja = nullptr, *Jb = nullptr, *r = nullptr;
    double *lstar = nullptr, *coef = nullptr, *rdiag = nullptr, *partial = nullptr;
    int partial_groups = 0;
    // plane dispatch order of the marches (c->g.zorder points here once set)
    int* zorder = nullptr;
    double* zscratch = nullptr;
    // FP32-sweep form: padded pair records {chi, S_hi} x 2 and their S_lo,
    // step offsets in those planes (poff32); double-float march: padded
    // {chi_hi, chi_lo, S_hi, S_lo} nodes and their step offsets (poff); both:
    // padded boundary B pairs; sum of the quadrature weights
    float4* pair = nullptr;
    float2* plo = nullptr;
    int* poff32 = nullptr;
    float4* node4 = nullptr;
    float2* b2 = nullptr;
    // LTE-diffusion inner boundary: dB/dtau of the bottom nodes (FP64, padded FP32)
    double* gdiff = nullptr;
    float* g2 = nullptr;
    bool gdiff_valid = false;
    // double-float march: df bilinear weights, df diffusion gradient
    float4* bwdf = nullptr;
    float2* g2df = nullptr;
    int* poff = nullptr;
    double wsum = 1.0;
    // direction tables
    DirInfo* info = nullptr;
    StepGeo* off = nullptr;
    Bw4d* bw = nullptr;
    Bw4d* bwh = nullptr;
    float4* bw32 = nullptr;
    double *d_mu = nullptr, *d_phi = nullptr, *d_w = nullptr;
    // scalars: [0] smax, [2] outer delta, [3] smallest source, [4] sweeps (d_sw)
    double* scal = nullptr;
    unsigned long long* d_steps = nullptr;
    double* h_scal = nullptr;               // pinned
    unsigned long long* h_steps = nullptr;  // pinned
    // per-sweep deltas of one Jacobi solve (device) and a pinned copy
    double* dlt = nullptr;
    double* h_dlt = nullptr;
    long long dlt_cap = 0;
    unsigned long long last_steps = 0;

    // Ng acceleration: period (0 = off), older iterates, reduction scratch
    int ng_period = 0;
    double ng_min_delta = 0.0;          // extrapolate only while the last delta >= this
    double ng_last_delta = 0.0;         // delta of the previous iteration
    int ng_count = 1;                   // iterates held, newest included
    double* ng_old[3] = {nullptr, nullptr, nullptr};  // J_{n-1}, J_{n-2}, J_{n-3}
    double* ng_part = nullptr;
    double* ng_out = nullptr;           // device [5]
    int ng_applied = 0;

    // profiling
    rt_stats stats{};
    bool profiling = false;
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};  // fs begin/end, jacobi begin/end
    bool fs_pending = false, jac_pending = false;

    std::string err;
};

namespace {

int fail(rt_ctx* c, int code, const char* fmt, ...)
{
    if (c) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof buf, fmt, ap);
        va_end(ap);
        c->err = buf;
    }
    return code;
}

#define CK(call)                                                                        \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return fail(c, e_ == cudaErrorMemoryAllocation ? RT_ENOMEM : RT_ECUDA,      \
                        "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    } while (0)

template <typename T>
void dfree(T*& p)
{
    if (p) cudaFree(p);
    p = nullptr;
}

template <typename T>
cudaError_t dalloc(T*& p, size_t count)
{
    dfree(p);
    if (count == 0) return cudaSuccess;
    return cudaMalloc((void**)&p, count * sizeof(T));
}

void free_ng(rt_ctx* c)
{
    for (auto& p : c->ng_old) dfree(p);
    dfree(c->ng_part);
    dfree(c->ng_out);
}

void free_os_graphs(rt_ctx* c)
{
    for (auto& e : c->osg) {
        if (e.exec) cudaGraphExecDestroy(e.exec);
        if (e.graph) cudaGraphDestroy(e.graph);
        e = rt_ctx::OsGraph{};
    }
}

// Working storage of the recording (freed with the grid or the directions).
void free_op_work(rt_ctx* c)
{
    dfree(c->ow_mem);
    c->ow_cap = 0;
    c->ow_ok = false;
    c->ow = rt_ctx::OpWork{};
    c->rec_valid = false;       // an operator's tables live there
}

void free_op_lists(rt_ctx* c)
{
    dfree(c->ol_mem);
    c->ol_cap = 0;
    c->ol_ok = false;
    c->ol = OpLists{};
}

void free_rec(rt_ctx* c)
{
    if (c->rec_mem) cudaFree(c->rec_mem);
    c->rec_mem = nullptr;
    c->rec = FsRec{};
    c->rec32 = Rec32{};
    c->op = OpMap{};
    c->rec_op = false;
    c->srec = nullptr;
    c->rec_cap = 0;
    c->rec_valid = false;
}

void free_grid_buffers(rt_ctx* c)
{
    free_os_graphs(c);
    dfree(c->chi); dfree(c->eps); dfree(c->B); dfree(c->J); dfree(c->S);
    dfree(c->Jfs); dfree(c->Jn); dfree(c->Ja); dfree(c->Jb); dfree(c->r);
    dfree(c->lstar); dfree(c->coef); dfree(c->rdiag); dfree(c->partial);
    dfree(c->node4); dfree(c->pair); dfree(c->plo);
    dfree(c->S_ref); dfree(c->J_ref); dfree(c->dS);
    dfree(c->b2); dfree(c->gdiff); dfree(c->g2); dfree(c->g2df);
    dfree(c->scpart); dfree(c->scplanes);
    dfree(c->zorder); dfree(c->zscratch);
    c->g.zorder = nullptr;
    c->scpart_n = c->scplanes_n = 0;
    free_ng(c);
    c->partial_groups = 0;
    free_rec(c);
    free_op_work(c);
    free_op_lists(c);
}

void free_tables(rt_ctx* c)
{
    dfree(c->info); dfree(c->off); dfree(c->bw); dfree(c->bwh); dfree(c->bw32);
    dfree(c->poff); dfree(c->poff32); dfree(c->bwdf);
    dfree(c->dn);
    dfree(c->d_mu); dfree(c->d_phi); dfree(c->d_w);
    c->ol_ok = c->ow_ok = c->rec_valid = false;     // made from them
}

// Add the device time of the kernels bracketed since the last harvest;
// called right after a stream synchronisation.
void harvest(rt_ctx* c)
{
    float ms = 0.f;
    if (c->fs_pending && cudaEventElapsedTime(&ms, c->ev[0], c->ev[1]) == cudaSuccess)
        c->stats.fs_ms += ms;
    if (c->jac_pending && cudaEventElapsedTime(&ms, c->ev[2], c->ev[3]) == cudaSuccess)
        c->stats.jacobi_ms += ms;
    c->fs_pending = c->jac_pending = false;
}

int enter(rt_ctx* c)
{
    if (!c) return RT_EINVAL;
    c->err.clear();
    cudaError_t e = cudaSetDevice(c->device);
    if (e != cudaSuccess) return fail(c, RT_ECUDA, "cudaSetDevice(%d): %s", c->device, cudaGetErrorString(e));
    return RT_OK;
}

// Default delta below which an RT_FP32_SWEEP solve continues in double-float
// (rt_set_df_finish): where the FP32 sweep's Ng extrapolation has to stop.
constexpr double kDefaultDfSwitch = 1e-6;

double default_cut(int precision)
{
    // FP32 sweep and double-float march: the cut is relative to S at the
    // voxel (see fs32.cu); 2^-46 (2^-52) keeps the truncation far below what
    // 1/eps can amplify at eps = 1e-6 (far below double-float rounding).
    if (precision == RT_FP64) return 1e-17;
    return precision == RT_DF64 ? 2.220446049250313e-16 : 1.4210854715202004e-14;
}

// Number of z-blocks that walk the kSlots direction slots: enough blocks to
// give every SM many waves, fewer (longer) blocks on large grids.
int auto_groups(const rt_ctx* c)
{
    if (c->groups_req > 0) return c->groups_req < kSlots ? c->groups_req : kSlots;
    const long long blocks = (long long)((c->g.nx * c->g.ny + 127) / 128) * c->g.nz;
    const long long target = 64LL * (c->num_sms > 0 ? c->num_sms : 152);
    int G = 1;
    while (G < kSlots && blocks * G < target) G *= 2;
    return G;
}

// The context's byte budget for a recording (rec_mode); 0 when the device
// cannot be asked.
long long rec_limit(const rt_ctx* c)
{
    if (c->rec_mode >= 0) return c->rec_mode;
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    // at most 60% of the device, leaving 2 GiB free
    const long long limit = (long long)(0.6 * (double)tot);
    const long long avail = (long long)fr + c->rec_cap - (2LL << 30);
    return avail < limit ? avail : limit;
}

// Device memory for a recording of `need` bytes within that budget: false
// when it does not fit or cannot be allocated.
bool rec_reserve(rt_ctx* c, long long need)
{
    if (need <= c->rec_cap) return true;
    if (need > rec_limit(c)) return false;
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) return false;
    free_rec(c);
    if (cudaMalloc((void**)&c->rec_mem, (size_t)need) != cudaSuccess) {
        cudaGetLastError();
        c->rec_mem = nullptr;
        return false;
    }
    c->rec_cap = need;
    return true;
}

long long up256(long long b) { return (b + 255) / 256 * 256; }

// Bytes a ray-by-ray recording of this context's march takes (0: its form
// does not record).
long long rec_need(const rt_ctx* c)
{
    if (c->fs_method != RT_FS_LONG || c->g.nz < 2 ||
        (c->src_order != RT_SRC_LINEAR && c->precision != RT_FP64))
        return 0;
    const long long tri = (long long)c->g.nz * (c->g.nz - 1) / 2;
    const long long b_slot = up256((long long)kSlots * c->g.N * (long long)sizeof(double));
    if (c->precision == RT_FP64 || c->precision == RT_DF64) {   // same bytes per entry
        const long long nxy = (long long)c->g.nx * c->g.ny, nwp = (nxy + 31) / 32;
        const long long b_cdn = c->src_order == RT_SRC_PARABOLIC
                                    ? up256((long long)c->g.ndir * c->g.N * (long long)sizeof(double))
                                    : 0;
        return up256((long long)c->g.ndir * nxy * tri * (long long)sizeof(double)) +
               up256((long long)c->g.ndir * c->g.nz * nwp * (long long)sizeof(int)) + 2 * b_slot +
               b_cdn;
    }
    const long long npair = (long long)c->g.nx * ((c->g.ny + 1) / 2), nwp = (npair + 31) / 32;
    return up256((long long)c->g.ndir * rec32_steps4(c->g.nz) * nwp * 32 * (long long)sizeof(float2)) +
           up256((long long)c->g.ndir * c->g.nz * nwp * (long long)sizeof(int)) + 2 * b_slot +
           up256(pair_records(c->g) * (long long)sizeof(float2));
}

// The ray-by-ray recording: whether this context records and replays its
// march (a form that records, within the byte budget), its buffers carved
// from one block.  When it does not fit, the march runs every time.
int ensure_rec(rt_ctx* c, bool& use)
{
    use = false;
    const long long need = rec_need(c);
    if (c->rec_mode == 0 || need == 0) return RT_OK;
    const long long tri = (long long)c->g.nz * (c->g.nz - 1) / 2;
    const long long b_slot = up256((long long)kSlots * c->g.N * (long long)sizeof(double));
    if (c->precision == RT_DF64) {
        const long long nxy = (long long)c->g.nx * c->g.ny;
        const long long nwp = (nxy + 31) / 32;
        const long long b_coef = up256((long long)c->g.ndir * nxy * tri * (long long)sizeof(float2));
        const long long b_lmax = up256((long long)c->g.ndir * c->g.nz * nwp * (long long)sizeof(int));
        if (!rec_reserve(c, need)) return RT_OK;
        c->rec32.coef = reinterpret_cast<float2*>(c->rec_mem);
        c->rec32.lmax = reinterpret_cast<int*>(c->rec_mem + b_coef);
        c->rec32.tsum = reinterpret_cast<double*>(c->rec_mem + b_coef + b_lmax);
        c->rec32.bc = reinterpret_cast<double*>(c->rec_mem + b_coef + b_lmax + b_slot);
        c->rec32.nwp = (int)nwp;
    } else if (c->precision == RT_FP64) {
        const long long nxy = (long long)c->g.nx * c->g.ny;
        const long long nwp = (nxy + 31) / 32;
        const long long b_coef = up256((long long)c->g.ndir * nxy * tri * (long long)sizeof(double));
        const long long b_lmax = up256((long long)c->g.ndir * c->g.nz * nwp * (long long)sizeof(int));
        if (!rec_reserve(c, need)) return RT_OK;
        c->rec.coef = reinterpret_cast<double*>(c->rec_mem);
        c->rec.lmax = reinterpret_cast<int*>(c->rec_mem + b_coef);
        c->rec.c0 = reinterpret_cast<double*>(c->rec_mem + b_coef + b_lmax);
        c->rec.bc = reinterpret_cast<double*>(c->rec_mem + b_coef + b_lmax + b_slot);
        c->rec.nwp = (int)nwp;
        const bool para = c->src_order == RT_SRC_PARABOLIC;
        c->rec.cdn = para ? reinterpret_cast<double*>(c->rec_mem + b_coef + b_lmax + 2 * b_slot)
                          : nullptr;
        c->rec.dn = para ? c->dn : nullptr;
    } else {
        const long long npair = (long long)c->g.nx * ((c->g.ny + 1) / 2);
        const long long nwp = (npair + 31) / 32;
        const long long b_coef = up256((long long)c->g.ndir * rec32_steps4(c->g.nz) * nwp * 32 *
                                       (long long)sizeof(float2));
        const long long b_lmax = up256((long long)c->g.ndir * c->g.nz * nwp * (long long)sizeof(int));
        const long long b_sp = up256(pair_records(c->g) * (long long)sizeof(float2));
        if (!rec_reserve(c, b_coef + b_lmax + 2 * b_slot + b_sp)) return RT_OK;
        char* q = c->rec_mem;
        c->rec32.coef = reinterpret_cast<float2*>(q);
        c->rec32.lmax = reinterpret_cast<int*>(q + b_coef);
        c->rec32.tsum = reinterpret_cast<double*>(q + b_coef + b_lmax);
        c->rec32.bc = reinterpret_cast<double*>(q + b_coef + b_lmax + b_slot);
        c->rec32.nwp = (int)nwp;
        c->srec = reinterpret_cast<float2*>(q + b_coef + b_lmax + 2 * b_slot);
    }
    use = true;
    return RT_OK;
}

// ---- assembled operator (op.cu) ------------------------------------------

// Grids and quadratures it handles: offsets in 31 bits, per-plane tables of
// 2 nz entries, a block's lengths in shared memory.
bool op_fits(const rt_ctx* c)
{
    return 4 * c->g.N < (1LL << 31) && c->g.nz <= 1024 && c->g.ndir <= 24 * 1024;
}

// The most entries and chunk rows the planes can have (every ray alive up
// to the boundary): eb, prow (exclusive prefix sums) and their totals.
void op_bounds(const rt_ctx* c, bool para, std::vector<long long>* eb, std::vector<long long>* prow,
               long long& entries, long long& rows)
{
    const long long nxy = (long long)c->g.nx * c->g.ny;
    const long long Dp = c->dpos, Dm = c->g.ndir - Dp;
    const long long up = std::min(nxy, 4 * Dp), um = std::min(nxy, 4 * Dm);
    const long long u2p = (up + 1) & ~1LL, u2m = (um + 1) & ~1LL;
    entries = rows = 0;
    for (int k = 0; k < c->g.nz; ++k) {
        const long long M = k, Mm = c->g.nz - 1 - k;
        if (eb) (*eb)[k] = entries;
        if (prow) (*prow)[k] = rows;
        long long e = M * u2p + Mm * u2m;
        if (para) e += (Mm > 0 ? u2p : 0) + (M > 0 ? u2m : 0);
        entries += (e + kOpPad - 1) / kOpPad * kOpPad;
        rows += Dp * M + Dm * Mm + (para ? c->g.ndir : 0);
    }
}

long long op_tiles(const rt_ctx* c) { return ((long long)c->g.nx * c->g.ny + 31) / 32; }

// Bytes of an operator of `entries` entries (its own terms included).
long long op_bytes(const rt_ctx* c, long long entries)
{
    return up256(entries * op_tiles(c) * 32 * (long long)sizeof(double)) +
           up256(entries * (long long)sizeof(int)) + 3 * up256(c->g.N * (long long)sizeof(double));
}

// Memory an operator may take: what the ray-by-ray recording takes and half as
// much again, at least 4 and at most 24 GiB (61 x 45 x 52 with 384 directions in
// double-float: 13 GB against 11.2).
long long op_budget(const rt_ctx* c, long long need)
{
    const long long extra = std::min(std::max(need / 2, 4LL << 30), 24LL << 30);
    return need + extra;
}

// Memory of the chunk buffer beside it: an eighth of the ray-by-ray recording, a
// chunk large enough to fill the GPU a few times over.  Where an operator near its
// budget left less, its planes were recorded a few at a time: first formal solution
// of 33^3 with 1024 directions through opaque spheres 34.2 ms in double-float and
// 55.0 in FP64, 15.5 and 44.9 with it.
long long op_chunk(long long need) { return std::max(need / 8, 2LL << 30); }

// Entries per recorded step up to which the operator is the faster form.  The
// entries of a plane are those of its longest rays, for all its voxels: where a
// medium is opaque but for a few columns they outnumber the steps, and the
// ray-by-ray replay does less.  45^3 x 256, operator over rays, formal solution and
// solve: slab with noise (2.8 entries per step) 0.53 and 0.67 in FP64, 0.59 and 0.71 in
// double-float; opaque with a column of 8% of the sides clear (6.9 and 7.2) 1.10
// and 1.01, 0.95 and 0.98; 10% (8.0 and 8.3) 1.25 and 1.11, 1.06 and 1.07; 25% (9.0 and
// 9.2) 1.41 and 1.53, 1.34 and 1.50; parabolic 7.1: 0.85 and 0.91, 8.8: 1.05 and 1.00.
double op_worth(const rt_ctx* c)
{
    return c->src_order == RT_SRC_PARABOLIC ? 8.5 : c->precision == RT_DF64 ? 7.5 : 7.0;
}

// The most memory a recording of this context asks for.
long long rec_ask(const rt_ctx* c, long long need)
{
    if (!op_fits(c)) return need;
    long long entries, rows;
    op_bounds(c, c->src_order == RT_SRC_PARABOLIC, nullptr, nullptr, entries, rows);
    const long long most = op_bytes(c, entries) +
                           up256(rows * c->g.nx * c->g.ny * (long long)sizeof(double));
    return std::max(need, std::min(most, op_budget(c, need) + op_chunk(need)));
}

// Bytes of a context's node lists and of its working storage.
long long op_list_bytes(const rt_ctx* c)
{
    const long long nxy = (long long)c->g.nx * c->g.ny, Q = 2LL * c->g.nz;
    const long long icap = 4LL * std::max(c->dpos, c->g.ndir - c->dpos), ucap = std::min(nxy, icap);
    return up256(4LL * c->g.ndir) + up256(4 * Q) + up256(4 * Q * ucap) + up256(4 * Q * (ucap + 1)) +
           up256(4 * Q * icap) + up256(4LL * c->g.ndir * c->g.nz) +
           up256((long long)sizeof(OpContrib) * Q * icap) + 256;
}

long long op_work_bytes(const rt_ctx* c)
{
    const long long T = (long long)c->g.ndir * c->g.nz, Q = 2LL * c->g.nz * c->g.nz;
    return up256(32 * c->g.N) + up256(4 * T * op_tiles(c)) + 3 * up256(4 * T) + 2 * up256(4 * Q) +
           4 * up256(8LL * c->g.nz) + 256 + 3 * up256(8LL * kSlots * c->g.N);
}

// A block of at least `need` bytes: the one that is there, unless it is too small or
// more than twice as large (a change of the quadrature that freed and allocated
// both blocks took 0.2 ms of the 0.38 of 20^3 with 8 directions).
cudaError_t keep_block(char*& mem, long long& cap, long long need)
{
    if (mem && cap >= need && cap <= 2 * need + (1LL << 20)) return cudaSuccess;
    dfree(mem);
    cap = 0;
    const cudaError_t e = cudaMalloc((void**)&mem, (size_t)need);
    if (e == cudaSuccess) cap = need;
    else mem = nullptr;
    return e;
}

// Node lists of the context's directions, built at the first recording.
int ensure_op_lists(rt_ctx* c)
{
    if (c->ol_ok) return RT_OK;
    const Geometry& g = c->g;
    const long long nxy = (long long)g.nx * g.ny, Q = 2LL * g.nz;
    const int Dmax = std::max(c->dpos, g.ndir - c->dpos);
    OpLists L{};
    L.dpos = c->dpos;
    L.icap = 4 * Dmax;
    L.ucap = (int)std::min(nxy, (long long)L.icap);
    const long long b_dord = up256(4LL * g.ndir), b_cnt = up256(4 * Q),
                    b_node = up256(4 * Q * L.ucap), b_start = up256(4 * Q * (L.ucap + 1)),
                    b_item = up256(4 * Q * L.icap), b_pos = up256(4LL * g.ndir * g.nz),
                    b_con = up256((long long)sizeof(OpContrib) * Q * L.icap);
    CK(keep_block(c->ol_mem, c->ol_cap, op_list_bytes(c)));
    char* q = c->ol_mem;
    int* dord = reinterpret_cast<int*>(q); q += b_dord;
    L.dord = dord;
    L.ucount = reinterpret_cast<int*>(q); q += b_cnt;
    L.unode = reinterpret_cast<int*>(q); q += b_node;
    L.ustart = reinterpret_cast<int*>(q); q += b_start;
    L.uofi = reinterpret_cast<int*>(q); q += b_item;
    L.posmax = reinterpret_cast<int*>(q); q += b_pos;
    L.contrib = reinterpret_cast<OpContrib*>(q); q += b_con;
    L.lpos = reinterpret_cast<int*>(q);
    int* scratch = nullptr;
    const long long ns = op_list_scratch(g);
    cudaError_t e = ns ? cudaMalloc((void**)&scratch, sizeof(int) * (size_t)ns) : cudaSuccess;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(dord, c->dord.data(), sizeof(int) * g.ndir, cudaMemcpyHostToDevice,
                            c->stream);
    if (e == cudaSuccess)
        e = launch_op_lists(g, c->info, c->off, c->bw, c->dn, L, scratch, c->stream);
    if (scratch) {
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
        cudaFree(scratch);
    }
    if (e != cudaSuccess) {
        free_op_lists(c);
        return fail(c, e == cudaErrorMemoryAllocation ? RT_ENOMEM : RT_ECUDA,
                    "building the operator's node lists: %s", cudaGetErrorString(e));
    }
    c->ol = L;
    c->ol_ok = true;
    c->stats.launches += 1;
    return RT_OK;
}

int ensure_op_work(rt_ctx* c)
{
    if (c->ow_ok) return RT_OK;
    const Geometry& g = c->g;
    const long long nwp = op_tiles(c), T = (long long)g.ndir * g.nz, Q = 2LL * g.nz * g.nz;
    const long long b_sp = up256(32 * g.N), b_lmax = up256(4 * T * nwp), b_t = up256(4 * T),
                    b_q = up256(4 * Q), b_z = up256(8LL * g.nz),
                    b_slot = up256(8LL * kSlots * g.N);
    CK(keep_block(c->ow_mem, c->ow_cap, op_work_bytes(c)));
    char* m = c->ow_mem;
    auto& w = c->ow;
    w.sp = reinterpret_cast<double*>(m); m += b_sp;
    w.lmax = reinterpret_cast<int*>(m); m += b_lmax;
    w.Lp = reinterpret_cast<int*>(m); m += b_t;
    w.rowbase = reinterpret_cast<int*>(m); m += b_t;
    w.poff = reinterpret_cast<int*>(m); m += b_t;
    w.cnt = reinterpret_cast<int*>(m); m += b_q;
    w.segb = reinterpret_cast<int*>(m); m += b_q;
    // (the host copies the steps, E and the rows together)
    w.steps = reinterpret_cast<unsigned long long*>(m); m += 256;
    w.E = reinterpret_cast<int*>(m); m += b_z;
    w.rows = reinterpret_cast<int*>(m); m += b_z;
    w.eb = reinterpret_cast<long long*>(m); m += b_z;
    w.prow = reinterpret_cast<long long*>(m); m += b_z;
    w.c0s = reinterpret_cast<double*>(m); m += b_slot;
    w.bcs = reinterpret_cast<double*>(m); m += b_slot;
    w.tss = reinterpret_cast<double*>(m);
    CK(launch_pad_offsets(g, c->info, c->off, 2LL * g.ny, w.poff, c->stream));
    c->ow_ok = true;
    c->ow_bounds = -1;
    c->stats.launches += 1;
    return RT_OK;
}

double cut_of(const rt_ctx* c);
ViewDF viewdf(rt_ctx* c);

// rc of an allocation that a recording can do without: no memory is no error.
bool no_memory(rt_ctx* c, int rc)
{
    if (rc != RT_ENOMEM) return false;
    c->err.clear();
    cudaGetLastError();
    return true;
}

// Below this bound on an operator's bytes its exact size is not asked for:
// the recording runs without a host wait.
constexpr long long kOpNoWait = 64LL << 20;

// Record the march of the current source (FP64, linear or parabolic, or
// double-float) and assemble its operator, or keep it ray by ray where the
// operator would take more memory (op_budget) or time (op_worth) or its lists get
// no memory.  use: whether a recording is held afterwards (not where the block or
// the working storage gets no memory: the march runs).
int ensure_op_rec(rt_ctx* c, int G, bool& use)
{
    use = false;
    const long long need = rec_need(c);
    if (c->rec_mode == 0 || need == 0) return RT_OK;
    if (c->rec_valid) {
        use = true;
        return RT_OK;
    }
    long long limit = std::max(rec_limit(c), c->rec_cap);
    if (need > limit) return RT_OK;
    int rc;
    if (!c->ow_ok) {
        if ((rc = ensure_op_work(c))) return no_memory(c, rc) ? RT_OK : rc;
        // what is left beside it
        limit = std::max(rec_limit(c), c->rec_cap);
        if (need > limit) {
            CK(cudaStreamSynchronize(c->stream));
            free_op_work(c);
            return RT_OK;
        }
    }
    const Geometry& g = c->g;
    const bool para = c->src_order == RT_SRC_PARABOLIC, df = c->precision == RT_DF64;
    const long long nxy = (long long)g.nx * g.ny, nwp = op_tiles(c);
    auto& w = c->ow;
    cudaStream_t st = c->stream;
    CK(launch_op_lengths(g, c->chi, c->S, c->scal + 0, c->info, w.poff, c->bw32,
                         cut_of(c) * kRecCutMargin, para ? kParaCutBits : df ? 1 : 0, df, G,
                         reinterpret_cast<float2*>(w.sp), w.lmax, (int)nwp, w.Lp, w.steps, st));
    c->stats.launches += 3;
    bool op = op_fits(c);
    std::vector<long long> eb(g.nz), prow(g.nz);
    std::vector<int> order(g.nz);
    for (int k = 0; k < g.nz; ++k) order[k] = k;
    std::vector<int> first{0, g.nz};    // ranks of the chunks' first planes
    long long entries = 0, rows = 0, chunk = 0;
    bool bounds = true;         // eb and prow are op_bounds'
    if (op && (rc = ensure_op_lists(c))) {
        if (!no_memory(c, rc)) return rc;
        op = false;
    }
    if (op) {
        CK(launch_op_counts(g, c->ol, para, w.Lp, w.rowbase, w.cnt, w.segb, w.E, w.rows, st));
        c->stats.launches += 1;
        op_bounds(c, para, &eb, &prow, entries, rows);
        chunk = up256(rows * nxy * (long long)sizeof(double));
        const long long room = std::max(std::min(limit, op_budget(c, need) + op_chunk(need)), c->rec_cap);
        if (op_bytes(c, entries) + chunk > std::min(room, kOpNoWait)) {
            bounds = false;
            // the size it really has, and chunks of planes
            const char* from = reinterpret_cast<const char*>(w.steps);
            std::vector<char> host(reinterpret_cast<const char*>(w.rows + g.nz) - from);
            CK(cudaMemcpyAsync(host.data(), from, host.size(), cudaMemcpyDeviceToHost, st));
            CK(cudaStreamSynchronize(st));
            c->stats.host_syncs += 1;
            unsigned long long steps;
            std::memcpy(&steps, host.data(), sizeof steps);
            const int* E = reinterpret_cast<const int*>(host.data() + (reinterpret_cast<const char*>(w.E) - from));
            const int* R = E + (w.rows - w.E);
            entries = rows = 0;
            long long most = 0;
            for (int k = 0; k < g.nz; ++k) {
                eb[k] = entries;
                entries += E[k];
                rows += R[k];
                most = std::max(most, (long long)R[k]);
            }
            const long long row = nxy * (long long)sizeof(double), own = op_bytes(c, entries);
            // a chunk as large as it should be, or the whole
            long long cb = std::min(rows, std::max(most, op_chunk(need) / row)) * row;
            if (own + up256(cb) > room) cb = std::max(most, rows / 12) * row;
            if (own + up256(cb) > room || own > op_budget(c, need) ||
                (double)entries * (double)(nwp * 32) > op_worth(c) * (double)steps) {
                op = false;
            } else {
                if (g.zorder && cb < rows * row) {
                    CK(cudaMemcpyAsync(order.data(), g.zorder, sizeof(int) * g.nz,
                                       cudaMemcpyDeviceToHost, st));
                    CK(cudaStreamSynchronize(st));
                    c->stats.host_syncs += 1;
                }
                first.assign(1, 0);
                long long at = 0;
                for (int r = 0; r < g.nz; ++r) {
                    if ((at + R[order[r]]) * row > cb) {
                        first.push_back(r);
                        at = 0;
                    }
                    prow[order[r]] = at;
                    at += R[order[r]];
                }
                first.push_back(g.nz);
                chunk = up256(cb);
            }
        }
    }
    if (op) {
        const long long own = op_bytes(c, entries);
        long long want = own + chunk;
        if (want > c->rec_cap) {
            // a little to spare, so that the next opacity fits as well
            const long long more = want + own / 64;
            if (!rec_reserve(c, more <= limit ? more : want)) op = false;
        }
    }
    if (!op) {
        if (!rec_reserve(c, need)) return RT_OK;
        if ((rc = ensure_rec(c, use))) return rc;
        if (!use) return RT_OK;
        CK(cudaMemcpyAsync(df ? c->rec32.lmax : c->rec.lmax, w.lmax, sizeof(int) * (size_t)g.ndir * g.nz * nwp,
                           cudaMemcpyDeviceToDevice, st));
    } else {
        const long long b_A = up256(entries * nwp * 32 * (long long)sizeof(double)),
                        b_off = up256(entries * (long long)sizeof(int)), b_n = up256(8 * g.N);
        char* q = c->rec_mem;
        c->op.A = reinterpret_cast<double*>(q); q += b_A;
        c->op.off = reinterpret_cast<int*>(q); q += b_off;
        c->op.c0 = reinterpret_cast<double*>(q); q += b_n;
        c->op.bc = reinterpret_cast<double*>(q); q += b_n;
        c->op.ts = reinterpret_cast<double*>(q);
        c->op.E = w.E;
        c->op.eb = w.eb;
        c->op.steps = w.steps;
        c->op.nwp = (int)nwp;
        // (the bounds depend on grid and directions only: copied once for them; two
        // copies of pageable memory take 7 of the 142 us of a first formal solution of 12^3)
        if (!bounds || c->ow_bounds != (para ? 1 : 0)) {
            CK(cudaMemcpyAsync(w.eb, eb.data(), sizeof(long long) * g.nz, cudaMemcpyHostToDevice, st));
            CK(cudaMemcpyAsync(w.prow, prow.data(), sizeof(long long) * g.nz, cudaMemcpyHostToDevice, st));
            c->ow_bounds = !bounds ? -1 : para ? 1 : 0;
        }
        CK(launch_op_offsets(g, c->ol, w.cnt, w.segb, c->op, st));
        c->stats.launches += 1;
    }
    RecOut ro{};
    ro.base = op ? reinterpret_cast<double*>(c->rec_mem + op_bytes(c, entries))  :
              df ? reinterpret_cast<double*>(c->rec32.coef) : c->rec.coef;
    ro.rowbase = op ? w.rowbase : nullptr;
    ro.prow = op ? w.prow : nullptr;
    ro.para = op && para ? 1 : 0;
    ro.cdn = op ? nullptr : c->rec.cdn;
    double* c0s = op ? w.c0s : df ? nullptr : c->rec.c0;
    double* bcs = op ? w.bcs : df ? c->rec32.bc : c->rec.bc;
    double* tss = op ? w.tss : c->rec32.tsum;
    for (size_t i = 0; i + 1 < first.size(); ++i) {
        const int r0 = first[i], np = first[i + 1] - r0;
        if (df)
            CK(launch_recdf(viewdf(c), r0, np, ro, w.lmax, (int)nwp, G, c0s, bcs, tss, st));
        else if (para)
            CK(launch_rec64p(g, r0, np, c->chi, c->B, c->gdiff, c->info, c->off, c->bw, c->bwh, c->dn,
                             ro, w.lmax, (int)nwp, G, c0s, bcs, st));
        else
            CK(launch_rec64(g, r0, np, c->chi, c->B, c->gdiff, c->info, c->off, c->bw, c->bwh, ro,
                            w.lmax, (int)nwp, G, c0s, bcs, st));
        c->stats.launches += 1;
        if (op) {
            CK(launch_op_assemble(g, df, r0, np, c->ol, ro, w.lmax, w.cnt, w.segb, c->op, st));
            c->stats.launches += 1;
        }
    }
    if (op) {
        CK(launch_op_own(g.N, w.c0s, w.bcs, df ? w.tss : nullptr, c->op, st));
        c->stats.launches += 1;
    }
    c->rec_op = op;
    c->op_steps = false;
    c->rec_valid = true;
    use = true;
    return RT_OK;
}

// Buffers of the short-characteristics march (sized by grid and directions).
int ensure_sc(rt_ctx* c)
{
    const size_t np = (size_t)sc_chunk(c->g) * (size_t)c->g.N;
    if (c->scpart_n < np) {
        dfree(c->scpart);
        c->scpart_n = 0;
        CK(dalloc(c->scpart, np));
        c->scpart_n = np;
    }
    const size_t ns = sc_scratch_planes(c->g);
    if (ns && c->scplanes_n < ns) {
        dfree(c->scplanes);
        c->scplanes_n = 0;
        CK(dalloc(c->scplanes, ns));
        c->scplanes_n = ns;
    }
    return RT_OK;
}

int ensure_partial(rt_ctx* c)
{
    if (c->partial_groups >= kSlots) return RT_OK;
    CK(dalloc(c->partial, (size_t)kSlots * c->g.N));
    c->partial_groups = kSlots;
    return RT_OK;
}

// Buffers the march of `precision` needs beyond the ones every form has:
// the FP32 pair planes, or the double-float nodes, gradient and weights
// (allocated once, also when a live context switches form).
int form_buffers(rt_ctx* c, int precision)
{
    if (c->have_grid && precision == RT_FP32_SWEEP && !c->pair) {
        CK(dalloc(c->pair, (size_t)pair_records(c->g)));
        CK(dalloc(c->plo, (size_t)pair_records(c->g)));
    }
    if (c->have_grid && precision == RT_DF64) {
        if (!c->node4) CK(dalloc(c->node4, (size_t)(4 * c->g.N)));
        if (!c->g2df) CK(dalloc(c->g2df, (size_t)4 * c->g.nx * c->g.ny));
    }
    if (c->have_quad && precision == RT_DF64 && !c->bwdf) {
        const long long T = (long long)c->g.ndir * c->g.nz;
        CK(dalloc(c->bwdf, (size_t)(2 * T)));
        CK(launch_bw_df(T, c->bw, c->bwdf, c->stream));
        c->stats.launches += 1;
    }
    return RT_OK;
}

int check_field(rt_ctx* c, const double* h, const char* what, bool positive, bool eps_range)
{
    for (long long v = 0; v < c->g.N; ++v) {
        const double x = h[v];
        if (!std::isfinite(x)) return fail(c, RT_EINVAL, "%s[%lld] is not finite", what, v);
        if (positive && !(x > 0)) return fail(c, RT_EINVAL, "%s[%lld] = %g must be > 0", what, v, x);
        if (eps_range && !(x > 0 && x <= 1))
            return fail(c, RT_EINVAL, "%s[%lld] = %g must lie in (0, 1]", what, v, x);
    }
    return RT_OK;
}

int need(rt_ctx* c, bool ok, const char* what)
{
    return ok ? RT_OK : fail(c, RT_ESTATE, "%s has not been set", what);
}

int need_all(rt_ctx* c)
{
    int rc;
    if ((rc = need(c, c->have_grid, "the grid"))) return rc;
    if ((rc = need(c, c->have_quad, "the quadrature"))) return rc;
    if ((rc = need(c, c->have_chi, "the opacity"))) return rc;
    if ((rc = need(c, c->have_eps, "epsilon"))) return rc;
    if ((rc = need(c, c->have_B, "the Planck function"))) return rc;
    return RT_OK;
}

cudaMemcpyKind kind(bool device) { return device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice; }

int set_field(rt_ctx* c, const double* src, double* dst, bool device, const char* what,
              bool positive, bool eps_range)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((rc = need(c, c->have_grid, "the grid"))) return rc;
    if (!src) return fail(c, RT_EINVAL, "%s is NULL", what);
    if (!device && (rc = check_field(c, src, what, positive, eps_range))) return rc;
    CK(cudaMemcpyAsync(dst, src, sizeof(double) * c->g.N, kind(device), c->stream));
    if (!device) CK(cudaStreamSynchronize(c->stream));
    return RT_OK;
}

View32 view32(rt_ctx* c)
{
    View32 v;
    v.g = c->g;
    v.pair = c->pair;
    v.lo = c->plo;
    v.b2 = c->b2;
    v.g2 = c->g2;
    v.info = c->info;
    v.off = c->off;
    v.poff = c->poff32;
    v.bw = c->bw32;
    v.smax = c->scal + 0;
    v.sfloor = nullptr;
    v.partial = c->partial;
    v.pmajor = plane_major32(c->g, c->order32);
    return v;
}

// The FP32 march of the finishing stage: source dS (packed in the pair
// planes), zero boundary intensities, cutoff relative to min |S_ref|.
View32 view32_fin(rt_ctx* c)
{
    View32 v = view32(c);
    v.g.top_bc = RT_BC_ZERO;
    v.g.bottom_bc = RT_BC_ZERO;
    v.sfloor = c->scal + 3;
    return v;
}

ViewDF viewdf(rt_ctx* c)
{
    ViewDF v;
    v.g = c->g;
    v.node = c->node4;
    v.b2 = c->b2;
    v.g2df = c->g2df;
    v.info = c->info;
    v.off = c->off;
    v.poff = c->poff;
    v.bw = c->bwdf;
    v.smax = c->scal + 0;
    v.partial = c->partial;
    return v;
}

// Formal solution: source in c->S (already set), result J into Jout (device).
// Pieces of one formal solution: per-problem preparation, the march itself,
// and the reduction over direction slots plus (once per opacity) Lambda*.
int fs_prepare(rt_ctx* c)
{
    int rc = ensure_partial(c);
    if (rc) return rc;
    if (c->g.bottom_bc == RT_BC_DIFFUSION && !c->gdiff_valid) {
        CK(launch_diffusion_grad(c->g, c->dz, c->chi, c->B, c->gdiff,
                                 c->precision == RT_FP32_SWEEP ? c->g2 : nullptr, c->stream));
        c->stats.launches += 1;
        if (c->precision == RT_DF64) {
            CK(launch_grad_df(c->g, c->gdiff, c->g2df, c->stream));
            c->stats.launches += 1;
        }
        c->gdiff_valid = true;
    }
    if (c->precision != RT_FP64 && !c->b2_valid) {
        CK(launch_pack_b2(c->g, c->B, c->b2, c->stream));
        c->b2_valid = true;
        c->stats.launches += 1;
    }
    return RT_OK;
}

double cut_of(const rt_ctx* c)
{
    return c->cut >= 0 ? c->cut : default_cut(c->precision);
}

// Lambda* is read off the operator (its own and nearest-node entries are the
// exact elements; 0.05 against 25 ms for the kernel on the 65^3 slab) unless
// the recording was cut so early that the cut shows in them.
constexpr double kOpLstarCut = 1e-15;

// direct: Jout holds J already (the assembled operator)
int fs_finish(rt_ctx* c, double* Jout, bool direct)
{
    if (direct) {
    } else if (c->precision == RT_FP64)
        CK(launch_sum_groups(c->g.N, c->partial, Jout, c->stream));
    else if (c->precision == RT_FP32_SWEEP && c->fin == 2)
        CK(launch_sum_groups_ref(c->g.N, c->partial, c->dS, c->wsum, c->J_ref, Jout, c->stream));
    else
        CK(launch_sum_groups_src(c->g.N, c->partial, c->S, c->wsum, Jout, c->stream));
    c->stats.launches += direct ? 0 : 1;
    if (!c->lstar_valid) {
        if (direct && cut_of(c) <= kOpLstarCut) {
            CK(launch_op_lstar(c->g, c->precision == RT_DF64, c->ol, c->op, c->ow.cnt, c->ow.segb, c->lstar, c->stream));
        } else if (c->src_order == RT_SRC_PARABOLIC) {
            CK(launch_lstar64p(c->g, c->chi, c->info, c->off, c->bw, c->dn, c->lstar, c->stream));
        } else if (c->precision == RT_FP64) {
            CK(launch_lstar64(c->g, c->chi, c->info, c->off, c->bw, c->lstar, c->stream));
        } else {
            // FP32 sweep and double-float march: Lambda* in double-float
            // (FP64-accurate; 5.7 against 25 ms for the FP64 kernel on the
            // 65^3 slab with 1024 directions), from the double-float nodes
            if (c->precision == RT_FP32_SWEEP) {
                int rc = form_buffers(c, RT_DF64);
                if (rc) return rc;
                CK(launch_packdf(c->g, c->chi, c->S, c->node4, c->stream));
                c->stats.launches += 1;
            }
            CK(launch_lstar_df(viewdf(c), false, c->lstar, c->stream));
        }
        c->lstar_valid = true;
        c->coef_valid = false;
        c->stats.launches += 1;
        c->stats.lstar_launches += 1;
    }
    return RT_OK;
}

// The finishing stage's reference (c->fin == 1): a double-float formal
// solution of the current source S into c->partial (same sum convention as
// the FP32 march); fin_record() then keeps S and J as the reference.
int fin_reference_march(rt_ctx* c, int G, unsigned long long* steps, cudaStream_t st)
{
    int rc = form_buffers(c, RT_DF64);
    if (rc) return rc;
    if (!c->S_ref) {
        CK(dalloc(c->S_ref, (size_t)c->g.N));
        CK(dalloc(c->J_ref, (size_t)c->g.N));
        CK(dalloc(c->dS, (size_t)c->g.N));
    }
    if (c->g.bottom_bc == RT_BC_DIFFUSION) {
        CK(launch_grad_df(c->g, c->gdiff, c->g2df, st));
        c->stats.launches += 1;
    }
    CK(launch_packdf(c->g, c->chi, c->S, c->node4, st));
    CK(launch_fsdf(viewdf(c), c->cut >= 0 ? c->cut : default_cut(RT_DF64), G, steps, st));
    c->stats.launches += 2;
    return RT_OK;
}

int fin_record(rt_ctx* c, const double* Jfs, cudaStream_t st)
{
    CK(cudaMemcpyAsync(c->S_ref, c->S, sizeof(double) * c->g.N, cudaMemcpyDeviceToDevice, st));
    CK(cudaMemcpyAsync(c->J_ref, Jfs, sizeof(double) * c->g.N, cudaMemcpyDeviceToDevice, st));
    CK(launch_absmin(c->g.N, c->S, c->scal + 3, st));
    c->stats.launches += 1;
    c->fin = 2;
    return RT_OK;
}

// Recorded short characteristics: the view, with the pairs of chi and S behind
// the weights in the recording's block.
ScView scview(rt_ctx* c)
{
    ScView v{};
    v.g = c->g;
    v.chi = c->chi;
    v.S = c->S;
    v.B = c->B;
    v.G = c->gdiff;
    v.info = c->info;
    v.off = c->off;
    v.bw = c->bw;
    v.bwdf = c->bwdf;
    if (c->precision == RT_DF64) {
        char* q = c->rec_mem + up256(sc_rec_bytes(c->g, true));
        v.chi2 = reinterpret_cast<const float2*>(q);
        v.S2 = reinterpret_cast<const float2*>(q + up256(8 * c->g.N));
    }
    return v;
}

// Record the weights of the short characteristics, once per opacity, where
// they fit the budget; use: whether they are held.
int ensure_sc_rec(rt_ctx* c, bool& use)
{
    use = false;
    if (c->rec_mode == 0) return RT_OK;
    const bool df = c->precision == RT_DF64;
    if (!c->rec_valid) {
        if (!rec_reserve(c, up256(sc_rec_bytes(c->g, df)) + (df ? 2 * up256(8 * c->g.N) : 0))) return RT_OK;
        const ScView v = scview(c);
        if (df) {
            CK(launch_sc_pairs(c->g.N, c->chi, const_cast<float2*>(v.chi2), c->stream));
            c->stats.launches += 1;
        }
        CK(launch_sc_record(v, df, c->rec_mem, c->stream));
        c->stats.launches += 1;
        c->rec_op = false;
        c->rec_valid = true;
    }
    use = true;
    return RT_OK;
}

// Short-characteristics formal solution: J straight from the march's ordered
// reduction, Lambda* from its own kernel once per opacity.
int run_fs_short(rt_ctx* c, double* Jout, bool count_steps)
{
    int rc = fs_prepare(c);
    if (rc) return rc;
    if ((rc = ensure_sc(c))) return rc;
    if (count_steps) CK(cudaMemsetAsync(c->d_steps, 0, sizeof(unsigned long long), c->stream));
    if (c->profiling) CK(cudaEventRecord(c->ev[0], c->stream));
    const bool df = c->precision == RT_DF64;
    bool use = false;
    if ((rc = ensure_sc_rec(c, use))) return rc;
    if (use) {
        const ScView v = scview(c);
        if (df) {
            CK(launch_sc_pairs(c->g.N, c->S, const_cast<float2*>(v.S2), c->stream));
            c->stats.launches += 1;
        }
        CK(launch_sc_apply(v, df, c->rec_mem, c->wsum, c->scpart, c->scplanes, Jout,
                           count_steps ? c->d_steps : nullptr, c->stream));
    } else if (df)
        CK(launch_scdf(viewdf(c), c->S, c->wsum, c->scpart, (float2*)c->scplanes, Jout,
                       count_steps ? c->d_steps : nullptr, c->stream));
    else
        CK(launch_sc64(c->g, c->chi, c->S, c->B, c->gdiff, c->info, c->off, c->bw, c->scpart,
                       c->scplanes, Jout, count_steps ? c->d_steps : nullptr, c->stream));
    if (c->profiling) {
        CK(cudaEventRecord(c->ev[1], c->stream));
        c->fs_pending = true;
    }
    const int chunks = (c->g.ndir + sc_chunk(c->g) - 1) / sc_chunk(c->g);
    c->stats.fs_launches += 1;
    c->stats.launches += 2 * chunks;
    if (!c->lstar_valid) {
        if (use)
            CK(launch_sc_lstar(scview(c), df, c->rec_mem, c->lstar, c->stream));
        else if (df)
            CK(launch_lstar_df(viewdf(c), true, c->lstar, c->stream));
        else
            CK(launch_lstar_sc64(c->g, c->chi, c->info, c->off, c->bw, c->lstar, c->stream));
        c->lstar_valid = true;
        c->coef_valid = false;
        c->stats.launches += 1;
        c->stats.lstar_launches += 1;
    }
    if (count_steps) {
        CK(cudaMemcpyAsync(c->h_steps, c->d_steps, sizeof(unsigned long long),
                           cudaMemcpyDeviceToHost, c->stream));
        c->op_steps = false;
    }
    return RT_OK;
}

// The formal solution comes from an operator that is there already.
bool op_ready(const rt_ctx* c)
{
    return (c->precision == RT_FP64 || c->precision == RT_DF64) && c->fs_method == RT_FS_LONG &&
           c->rec_mode != 0 && c->rec_valid && c->rec_op;
}

// The FP32 sweep replays a recording that is there already (the finishing
// stage's reference marches).
bool rep_ready(const rt_ctx* c)
{
    return c->precision == RT_FP32_SWEEP && c->fs_method == RT_FS_LONG && c->rec_mode != 0 && c->rec_valid &&
           c->fin != 1;
}

// The source records of the replay, where prepare_source has not formed them
// (the recording was made in between, from S).
int rep_source(rt_ctx* c)
{
    if (!c->op_packed) {
        CK(launch_pack_srecs(c->g, c->S, nullptr, nullptr, nullptr, nullptr, nullptr, c->srec, c->stream));
        c->stats.launches += 1;
    }
    c->op_packed = false;
    return RT_OK;
}

// The source packed for the operator, where prepare_source has not (the
// operator was made in between).
int op_source(rt_ctx* c)
{
    if (!c->op_packed) {
        CK(launch_op_pack(c->g, c->S, nullptr, nullptr, nullptr, c->precision == RT_DF64, c->ow.sp, c->stream));
        c->stats.launches += 1;
    }
    c->op_packed = false;
    return RT_OK;
}

// The double-float formal solution of a context: recorded in the first one
// after the opacities change and replayed, or marched when the recording
// does not fit.  direct: J is in Jout, else in the slots of c->partial.
int df_formal(rt_ctx* c, int G, double* Jout, unsigned long long* steps, bool& direct)
{
    bool use = false;
    int rc = ensure_op_rec(c, G, use);
    if (rc) return rc;
    direct = use && c->rec_op;
    if (direct) {
        if ((rc = op_source(c))) return rc;
        CK(launch_op_apply_df(c->g, c->S, c->ow.sp, c->op, c->wsum, Jout, steps, c->stream));
        c->stats.launches += 1;
    } else if (use) {
        CK(launch_fsdfrep(viewdf(c), c->rec32, G, steps, c->stream));
    } else {
        CK(launch_fsdf(viewdf(c), cut_of(c), G, steps, c->stream));
    }
    return RT_OK;
}

// The FP64 formal solution of a context: recorded in the first one after
// the opacities, directions or boundary change (J then comes from the
// recording like every later one, so that it does not depend on which
// formal solution recorded), or marched when the recording does not fit.
// direct: J is in Jout, else in the slots of c->partial.
int fs64_formal(rt_ctx* c, int G, double* Jout, unsigned long long* steps, bool& direct)
{
    bool use = false;
    int rc = ensure_op_rec(c, G, use);
    if (rc) return rc;
    direct = use && c->rec_op;
    cudaStream_t st = c->stream;
    if (direct) {
        if ((rc = op_source(c))) return rc;
        CK(launch_op_apply64(c->g, c->S, c->ow.sp, c->op, Jout, steps, st));
        c->stats.launches += 1;
    } else if (use) {
        CK(launch_fs64rep(c->g, c->S, c->info, c->off, c->bw, c->rec, G, c->partial, steps, st));
    } else if (c->src_order == RT_SRC_PARABOLIC) {
        CK(launch_fs64p(c->g, c->chi, c->S, c->B, c->gdiff, c->info, c->off, c->bw, c->dn,
                        c->scal + 0, cut_of(c), G, c->partial, steps, st));
    } else {
        CK(launch_fs64(c->g, c->chi, c->S, c->B, c->gdiff, c->info, c->off, c->bw, c->bwh,
                       c->scal + 0, cut_of(c), G, c->partial, steps, st));
    }
    return RT_OK;
}

int run_fs(rt_ctx* c, double* Jout, bool count_steps)
{
    if (c->fs_method == RT_FS_SHORT) return run_fs_short(c, Jout, count_steps);
    const int G = auto_groups(c);
    int rc = fs_prepare(c);
    if (rc) return rc;
    // an operator's steps are those of its recording: counted once
    count_steps = count_steps && !(op_ready(c) && c->op_steps);
    if (count_steps) CK(cudaMemsetAsync(c->d_steps, 0, sizeof(unsigned long long), c->stream));
    const double cut = cut_of(c);
    if (c->profiling) CK(cudaEventRecord(c->ev[0], c->stream));
    bool direct = false;
    if (c->precision == RT_FP64) {
        if ((rc = fs64_formal(c, G, Jout, count_steps ? c->d_steps : nullptr, direct))) return rc;
    } else if (c->precision == RT_DF64) {
        if ((rc = df_formal(c, G, Jout, count_steps ? c->d_steps : nullptr, direct))) return rc;
    } else if (c->fin == 1) {
        if ((rc = fin_reference_march(c, G, count_steps ? c->d_steps : nullptr, c->stream)))
            return rc;
    } else {
        // FP32 sweep (fin 0, or 2: the finishing stage's source change).  The
        // recording is made from the source itself (fin 0) and serves both.
        bool use = false;
        if ((rc = ensure_rec(c, use))) return rc;
        unsigned long long* sp = count_steps ? c->d_steps : nullptr;
        if (use && !c->rec_valid && c->fin == 0) {
            CK(launch_fs32rec(view32(c), cut * kRecCutMargin, G, c->rec32, sp, c->stream));
            c->rec_valid = true;
            c->stats.launches += 1;
        }
        if (use && c->rec_valid) {
            if ((rc = rep_source(c))) return rc;
            Rep32 rp{c->g, c->srec, c->info, c->poff32, c->bw32, c->rec32, c->partial,
                     c->fin == 2 ? 1 : 0, plane_major32(c->g, c->order32)};
            CK(launch_fs32rep(rp, G, c->threads32, sp, c->stream));
            c->stats.launches += 1;
        } else {
            CK(launch_fs32d(c->fin == 2 ? view32_fin(c) : view32(c), cut, G, c->threads32, sp,
                            c->stream));
        }
    }
    if (c->profiling) {
        CK(cudaEventRecord(c->ev[1], c->stream));
        c->fs_pending = true;
    }
    c->stats.fs_launches += 1;
    c->stats.launches += 1;
    if ((rc = fs_finish(c, Jout, direct))) return rc;
    if (c->precision == RT_FP32_SWEEP && c->fin == 1 && (rc = fin_record(c, Jout, c->stream)))
        return rc;
    if (count_steps) {
        CK(cudaMemcpyAsync(c->h_steps, c->d_steps, sizeof(unsigned long long),
                           cudaMemcpyDeviceToHost, c->stream));
        c->op_steps = direct;
    }
    return RT_OK;
}

// S = eps B + (1 - eps) J (or the caller's S), then in the form of the next
// formal solution: packed for the operator or the replay (whose cutoffs are
// made: no smax), else (march: always) smax and the FP32 or double-float records.
int prepare_source(rt_ctx* c, const double* S_in, bool device, bool march)
{
    c->op_packed = !march && op_ready(c);
    if (!march && rep_ready(c)) {
        if (S_in)
            CK(cudaMemcpyAsync(c->S, S_in, sizeof(double) * c->g.N, kind(device), c->stream));
        CK(launch_pack_srecs(c->g, c->S, S_in ? nullptr : c->eps, c->B, c->J,
                             c->fin == 2 ? c->S_ref : nullptr, c->dS, c->srec, c->stream));
        c->stats.launches += 1;
        c->op_packed = true;
        return RT_OK;
    }
    if (c->op_packed) {
        if (S_in)
            CK(cudaMemcpyAsync(c->S, S_in, sizeof(double) * c->g.N, kind(device), c->stream));
        CK(launch_op_pack(c->g, c->S, S_in ? nullptr : c->eps, c->B, c->J, c->precision == RT_DF64, c->ow.sp,
                          c->stream));
        c->stats.launches += 1;
        return RT_OK;
    }
    const bool bnd = c->g.top_bc || c->g.bottom_bc;
    CK(cudaMemsetAsync(c->scal + 0, 0, sizeof(double), c->stream));
    if (S_in) {
        CK(cudaMemcpyAsync(c->S, S_in, sizeof(double) * c->g.N, kind(device), c->stream));
        CK(launch_absmax(c->g.N, c->S, bnd ? c->B : nullptr, c->scal + 0, nullptr, c->stream));
    } else {
        CK(launch_source(c->g.N, c->eps, c->B, c->J, c->S, nullptr, bnd ? c->B : nullptr,
                         c->scal + 0, c->stream));
    }
    c->stats.launches += 1;
    if (c->precision == RT_FP32_SWEEP && c->fin == 2) {
        // finishing stage: march dS = S - S_ref, cutoff bound max |dS|
        CK(launch_delta_source(c->g.N, c->S, c->S_ref, c->dS, c->stream));
        CK(cudaMemsetAsync(c->scal + 0, 0, sizeof(double), c->stream));
        CK(launch_absmax(c->g.N, c->dS, nullptr, c->scal + 0, nullptr, c->stream));
        CK(launch_pack_pairs(c->g, c->chi, c->dS, c->pair, c->plo, c->stream));
        c->stats.launches += 3;
    } else if (c->precision == RT_FP32_SWEEP && c->fin == 1) {
        // the reference formal solution packs its own double-float nodes
    } else if (c->precision == RT_FP32_SWEEP) {
        CK(launch_pack_pairs(c->g, c->chi, c->S, c->pair, c->plo, c->stream));
        c->stats.launches += 1;
    } else if (c->precision == RT_DF64 && c->rec_valid && c->fs_method == RT_FS_SHORT) {
        // the recorded short characteristics pack their own
    } else if (c->precision == RT_DF64) {
        CK(launch_packdf(c->g, c->chi, c->S, c->node4, c->stream));
        c->stats.launches += 1;
    }
    return RT_OK;
}

// Checked builds: report (and clear) the first out-of-bounds index the
// kernels recorded since the last check.  Normal builds: nothing to do.
int check_bounds(rt_ctx* c, int rc)
{
#ifdef RT_CHECKED
    unsigned long long h[4] = {0, 0, 0, 0};
    if (cudaMemcpy(h, c->berr, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess)
        return fail(c, RT_ECUDA, "reading the bounds record failed");
    if (h[0]) {
        cudaMemset(c->berr, 0, sizeof(h));
        return fail(c, RT_EBOUNDS, "index %lld outside [0, %lld) at site %llu",
                    (long long)h[2], (long long)h[3], h[1]);
    }
#else
    (void)c;
#endif
    return rc;
}

int formal_solution(rt_ctx* c, const double* S, double* Jfs_out, double* lstar_out, bool device)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((rc = need_all(c))) return rc;
    if (!Jfs_out) return fail(c, RT_EINVAL, "J_fs is NULL");
    if ((rc = prepare_source(c, S, device, false))) return rc;
    if ((rc = run_fs(c, c->Jfs, true))) return rc;
    const cudaMemcpyKind out = device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    CK(cudaMemcpyAsync(Jfs_out, c->Jfs, sizeof(double) * c->g.N, out, c->stream));
    if (lstar_out)
        CK(cudaMemcpyAsync(lstar_out, c->lstar, sizeof(double) * 27 * c->g.N, out, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    harvest(c);
    c->last_steps = *c->h_steps;
    c->stats.steps += c->last_steps;
    return RT_OK;
}

int ensure_coef(rt_ctx* c)
{
    if (c->coef_valid) return RT_OK;
    CK(launch_os_coef(c->g, c->lstar, c->eps, c->coef, c->rdiag,
                      c->os_method == RT_OS_GAUSS_SEIDEL, c->stream));
    c->coef_valid = true;
    c->stats.launches += 1;
    return RT_OK;
}

int ensure_dlt(rt_ctx* c, long long max_sweeps)
{
    if (c->dlt_cap >= max_sweeps) return RT_OK;
    const long long cap = std::max(max_sweeps, 1024LL);
    free_os_graphs(c);          // they hold the old dlt pointer
    c->dlt_cap = 0;
    CK(dalloc(c->dlt, (size_t)cap));
    if (c->h_dlt) cudaFreeHost(c->h_dlt);
    c->h_dlt = nullptr;
    CK(cudaMallocHost((void**)&c->h_dlt, sizeof(double) * cap));
    c->dlt_cap = cap;
    return RT_OK;
}

// Jacobi solve from J_old (device) into J_new (device); J_fs device.  Sweeps
// are enqueued in growing chunks; a sweep that follows a converged one is a
// no-op on the device, so checking once per chunk gives exactly the sweeps
// of a check after every sweep.
// The operator-splitting step as one CUDA graph: right-hand side, zeroed
// deltas, J_old copied to the sweep buffer read first, a zeroed sweep
// counter, then a WHILE node whose body runs two sweeps and the loop test on
// the device.  The host launches it once and reads the deltas once, instead
// of synchronising after every chunk of sweeps.  Results are those of the
// host loop: same kernels, same no-op rule after convergence.
int build_os_graph(rt_ctx* c, rt_ctx::OsGraph& e, const double* Jfs, const double* Jold,
                   double* Jnew, double tol, int max_sweeps)
{
    const bool gs = c->os_method == RT_OS_GAUSS_SEIDEL;
    cudaGraph_t g = nullptr;
    CK(cudaGraphCreate(&g, 0));
    cudaGraphConditionalHandle h;
    cudaError_t err = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault);
    std::vector<cudaGraphNode_t> deps;
    if (err == cudaSuccess)
        err = cudaStreamBeginCaptureToGraph(c->stream, g, nullptr, nullptr, 0,
                                            cudaStreamCaptureModeThreadLocal);
    if (err == cudaSuccess) {
        // prologue; every call is attempted so that the capture is always ended
        cudaError_t e1 = launch_os_rhs(c->g, c->coef, c->rdiag, Jfs, Jold, c->r, gs, c->stream);
        cudaError_t e2 = cudaMemsetAsync(c->dlt, 0, sizeof(double) * ((size_t)max_sweeps + kPassSweeps), c->stream);
        cudaError_t e3 = cudaMemcpyAsync(c->Jb, Jold, sizeof(double) * c->g.N,
                                         cudaMemcpyDeviceToDevice, c->stream);
        cudaError_t e4 = cudaMemsetAsync(c->d_nsw, 0, sizeof(int), c->stream);
        cudaStreamCaptureStatus cs;
        const cudaGraphNode_t* dp = nullptr;
        size_t nd = 0;
        cudaError_t e5 = cudaStreamGetCaptureInfo(c->stream, &cs, nullptr, nullptr, &dp, nullptr, &nd);
        if (e5 == cudaSuccess) deps.assign(dp, dp + nd);
        cudaGraph_t out = nullptr;
        cudaError_t e6 = cudaStreamEndCapture(c->stream, &out);
        for (cudaError_t x : {e1, e2, e3, e4, e5, e6})
            if (err == cudaSuccess && x != cudaSuccess) err = x;
    }
    cudaGraphNodeParams cp = {};
    cudaGraphNode_t cn;
    if (err == cudaSuccess) {
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        err = cudaGraphAddNode(&cn, g, deps.data(), nullptr, deps.size(), &cp);
    }
    if (err == cudaSuccess) {
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        err = cudaStreamBeginCaptureToGraph(c->stream, body, nullptr, nullptr, 0,
                                            cudaStreamCaptureModeThreadLocal);
        if (err == cudaSuccess) {
            cudaError_t e1 = launch_sweep_pass(c->g, c->coef, c->r, c->Ja, c->Jb, c->dlt, c->d_nsw,
                                               max_sweeps, tol, gs, h, c->stream);
            cudaGraph_t out = nullptr;
            cudaError_t e2 = cudaStreamEndCapture(c->stream, &out);
            err = e1 != cudaSuccess ? e1 : e2;
        }
    }
    if (err == cudaSuccess) {
        // epilogue after the loop: the last sweep's iterate into J_new and
        // the sweep count, on the device
        err = cudaStreamBeginCaptureToGraph(c->stream, g, &cn, nullptr, 1,
                                            cudaStreamCaptureModeThreadLocal);
        if (err == cudaSuccess) {
            cudaError_t e1 = launch_os_select(c->g.N, c->dlt, max_sweeps, tol, c->Ja, c->Jb, Jnew,
                                              c->d_sw, c->stream);
            cudaGraph_t out = nullptr;
            cudaError_t e2 = cudaStreamEndCapture(c->stream, &out);
            err = e1 != cudaSuccess ? e1 : e2;
        }
    }
    cudaGraphExec_t exec = nullptr;
    if (err == cudaSuccess) err = cudaGraphInstantiate(&exec, g, 0);
    if (err != cudaSuccess) {
        cudaGraphDestroy(g);
        cudaGetLastError();
        return fail(c, RT_ECUDA, "building the operator-splitting graph: %s", cudaGetErrorString(err));
    }
    e.graph = g;
    e.exec = exec;
    e.jold = Jold;
    e.jfs = Jfs;
    e.jnew = Jnew;
    e.dlt = c->dlt;
    e.max_sweeps = max_sweeps;
    e.method = c->os_method;
    e.tol = tol;
    return RT_OK;
}

int ensure_sweep_words(rt_ctx* c);

// The operator-splitting step as one graph launch, without waiting for it:
// J_new and the sweep count (c->d_sw) are written on the device.  The
// caller copies d_sw to h_sw before its next synchronisation and then calls
// os_graph_done().
int run_os_graph(rt_ctx* c, const double* Jfs, const double* Jold, double* Jnew, double tol_inner,
                 int max_sweeps)
{
    int rc;
    if ((rc = ensure_dlt(c, (long long)max_sweeps + kPassSweeps)) || (rc = ensure_sweep_words(c))) return rc;
    c->os_one = false;
    rt_ctx::OsGraph* e = nullptr;
    for (auto& x : c->osg)
        if (x.exec && x.jold == Jold && x.jfs == Jfs && x.jnew == Jnew && x.dlt == c->dlt &&
            x.max_sweeps == max_sweeps && x.tol == tol_inner && x.method == c->os_method)
            e = &x;
    if (!e) {
        e = &c->osg[c->osg_next];
        c->osg_next ^= 1;
        if (e->exec) cudaGraphExecDestroy(e->exec);
        if (e->graph) cudaGraphDestroy(e->graph);
        *e = rt_ctx::OsGraph{};
        if ((rc = build_os_graph(c, *e, Jfs, Jold, Jnew, tol_inner, max_sweeps))) return rc;
    }
    if (c->profiling) CK(cudaEventRecord(c->ev[2], c->stream));
    CK(cudaGraphLaunch(e->exec, c->stream));
    if (c->profiling) {
        CK(cudaEventRecord(c->ev[3], c->stream));
        c->jac_pending = true;
    }
    CK(cudaMemcpyAsync(c->h_sw, c->d_sw, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    return RT_OK;
}

// After the synchronisation that follows run_os_graph or run_os_one: the
// sweep count into *sweeps, and the counters of that step.
int os_graph_done(rt_ctx* c, int* sweeps)
{
    *sweeps = *c->h_sw;
    if (*sweeps < 0)
        return fail(c, RT_ETIMEOUT, "a wait of the operator-splitting kernel's blocks gave up");
    const int per = c->os_method == RT_OS_GAUSS_SEIDEL ? 2 : 1;
    const int passes = (*sweeps + kPassSweeps - 1) / kPassSweeps;
    c->stats.launches += c->os_one ? 1 : 2 + passes * (kPassSweeps * per + 1);
    c->stats.jacobi_launches += c->os_one ? *sweeps * per : passes * kPassSweeps * per;
    return RT_OK;
}

// Barrier words that the one-kernel solves use at most (of a set; of all problems
// of a batch): 32 MB.  Above them the sweeps run as a graph, which needs a word per sweep too
// but does not zero them in a kernel of few blocks.
constexpr long long kBarWords = 1LL << 22;

// Barriers of a solve.
long long os_barriers(const rt_ctx* c, int max_sweeps)
{
    return (long long)max_sweeps * (c->os_method == RT_OS_GAUSS_SEIDEL ? 2 : 1);
}

// Two sets of at least `words` zeroed barrier words (the set in turn).
int ensure_os_words(rt_ctx* c, int words)
{
    if (c->os_cap >= words) return RT_OK;
    const int cap = std::max(words, 1024);
    c->os_cap = 0;
    CK(dalloc(c->os_words, 2 * (size_t)cap));
    CK(cudaMemsetAsync(c->os_words, 0, sizeof(unsigned long long) * 2 * cap, c->stream));
    c->os_cap = cap;
    c->os_dirty[0] = c->os_dirty[1] = 0;
    return RT_OK;
}

// The context's arrays as a task of launch_os_solve.
OsTask os_task(const rt_ctx* c, const double* Jfs, const double* Jold, double* Jnew,
               unsigned long long* words, int* sweeps, int nblk)
{
    OsTask t;
    t.g = c->g;
    t.c = c->coef;
    t.rdiag = c->rdiag;
    t.Jfs = Jfs;
    t.Jold = Jold;
    t.Ja = c->Ja;
    t.Jb = c->Jb;
    t.Jn = Jnew;
    t.words = words;
    t.clear = nullptr;
    t.nclear = 0;
    t.zero = nullptr;
    t.delta = c->os_delta;
    t.hist = c->os_hist;
    t.sweeps = sweeps;
    t.nblk = nblk;
    return t;
}

int ensure_sweep_words(rt_ctx* c)
{
    if (!c->d_nsw) CK(cudaMalloc((void**)&c->d_nsw, sizeof(int)));
    return RT_OK;
}

// The operator-splitting step as one cooperative kernel, without waiting for
// it, where the grid's blocks are resident together; ran: whether it was
// launched.  In a solve it zeroes the outer delta, and the caller copies that
// and the sweep count back together.
int run_os_one(rt_ctx* c, const double* Jfs, const double* Jold, double* Jnew, double tol_inner,
               int max_sweeps, bool in_solve, bool& ran)
{
    ran = false;
    OsShape sh;
    os_solve_shape(c->g.N, c->num_sms, c->os_method == RT_OS_GAUSS_SEIDEL, &sh);
    if (sh.blocks == 0) return RT_OK;
    if (os_barriers(c, max_sweeps) > kBarWords) return RT_OK;
    int rc;
    const int words = (int)os_barriers(c, max_sweeps);
    if ((rc = ensure_os_words(c, words))) return rc;
    const int set = c->os_set;
    OsTask t = os_task(c, Jfs, Jold, Jnew, c->os_words + (long long)set * c->os_cap, c->d_sw, sh.blocks);
    t.clear = c->os_words + (long long)(set ^ 1) * c->os_cap;
    t.nclear = c->os_dirty[set ^ 1];
    if (in_solve) t.zero = c->scal + 2;
    if (c->profiling) CK(cudaEventRecord(c->ev[2], c->stream));
    const cudaError_t e = launch_os_solve(t, nullptr, nullptr, 1, sh, c->os_method == RT_OS_GAUSS_SEIDEL,
                                          c->num_sms, max_sweeps, tol_inner, c->stream);
    if (e == cudaErrorCooperativeLaunchTooLarge) return RT_OK;
    CK(e);
    c->os_dirty[set ^ 1] = 0;
    c->os_dirty[set] = words;
    c->os_set = set ^ 1;
    if (c->profiling) {
        CK(cudaEventRecord(c->ev[3], c->stream));
        c->jac_pending = true;
    }
    if (!in_solve)
        CK(cudaMemcpyAsync(c->h_sw, c->d_sw, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    c->os_one = ran = true;
    return RT_OK;
}

int run_os(rt_ctx* c, const double* Jfs, const double* Jold, double* Jnew, double tol_inner,
           int max_sweeps, bool in_solve, int* sweeps_out)
{
    c->os_one = false;
    int rc = ensure_coef(c);
    if (rc) return rc;
    if (c->use_graphs) {
        // sweep count after the caller's synchronisation (os_graph_done)
        if (sweeps_out) *sweeps_out = -1;
        bool ran = false;
        if ((rc = run_os_one(c, Jfs, Jold, Jnew, tol_inner, max_sweeps, in_solve, ran)) || ran)
            return rc;
        return run_os_graph(c, Jfs, Jold, Jnew, tol_inner, max_sweeps);
    }
    if ((rc = ensure_dlt(c, max_sweeps))) return rc;
    const bool gs = c->os_method == RT_OS_GAUSS_SEIDEL;
    CK(launch_os_rhs(c->g, c->coef, c->rdiag, Jfs, Jold, c->r, gs, c->stream));
    c->stats.launches += 1;
    CK(cudaMemsetAsync(c->dlt, 0, sizeof(double) * max_sweeps, c->stream));
    double* bufs[2] = {c->Ja, c->Jb};
    int launched = 0, done = -1, chunk = 2;
    while (launched < max_sweeps && done < 0) {
        const int n0 = launched;
        const int n1 = launched + chunk < max_sweeps ? launched + chunk : max_sweeps;
        if (c->profiling) CK(cudaEventRecord(c->ev[2], c->stream));
        for (int n = n0; n < n1; ++n) {
            const double* cur = n == 0 ? Jold : bufs[(n - 1) & 1];
            if (gs)
                CK(launch_gs_sweep(c->g, c->coef, c->r, cur, bufs[n & 1], c->dlt, n, tol_inner,
                                   c->stream));
            else
                CK(launch_jacobi(c->g, c->coef, c->r, cur, bufs[n & 1], c->dlt, n, tol_inner,
                                 c->stream));
        }
        if (c->profiling) {
            CK(cudaEventRecord(c->ev[3], c->stream));
            c->jac_pending = true;
        }
        c->stats.launches += (gs ? 2 : 1) * (n1 - n0);
        c->stats.jacobi_launches += (gs ? 2 : 1) * (n1 - n0);
        CK(cudaMemcpyAsync(c->h_dlt + n0, c->dlt + n0, sizeof(double) * (n1 - n0),
                           cudaMemcpyDeviceToHost, c->stream));
        CK(cudaStreamSynchronize(c->stream));
        c->stats.host_syncs += 1;
        harvest(c);
        for (int n = n0; n < n1; ++n)
            if (c->h_dlt[n] < tol_inner) {
                done = n;
                break;
            }
        launched = n1;
        if (chunk < 32) chunk *= 2;
    }
    const int sweeps = done >= 0 ? done + 1 : max_sweeps;
    CK(cudaMemcpyAsync(Jnew, bufs[(sweeps - 1) & 1], sizeof(double) * c->g.N,
                       cudaMemcpyDeviceToDevice, c->stream));
    if (sweeps_out) *sweeps_out = sweeps;
    return RT_OK;
}

int os_step(rt_ctx* c, const double* Jfs, const double* Jold, double* Jnew, double tol_inner,
            int max_sweeps, int* sweeps, bool device)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((rc = need_all(c))) return rc;
    if (!c->lstar_valid) return fail(c, RT_ESTATE, "Lambda* is not built: run a formal solution first");
    if (!Jfs || !Jold || !Jnew) return fail(c, RT_EINVAL, "null J pointer");
    if (max_sweeps < 1) return fail(c, RT_EINVAL, "max_sweeps must be >= 1");
    const double* dfs = Jfs;
    const double* dold = Jold;
    if (!device) {
        CK(cudaMemcpyAsync(c->Jfs, Jfs, sizeof(double) * c->g.N, cudaMemcpyHostToDevice, c->stream));
        CK(cudaMemcpyAsync(c->Jn, Jold, sizeof(double) * c->g.N, cudaMemcpyHostToDevice, c->stream));
        dfs = c->Jfs;
        dold = c->Jn;
    }
    double* dnew = device ? Jnew : c->S;  // S is free as scratch here
    int ns = 0;
    if ((rc = run_os(c, dfs, dold, dnew, tol_inner, max_sweeps, false, &ns))) return rc;
    if (!device)
        CK(cudaMemcpyAsync(Jnew, dnew, sizeof(double) * c->g.N, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    harvest(c);
    if (ns < 0 && (rc = os_graph_done(c, &ns))) return rc;
    if (sweeps) *sweeps = ns;
    return RT_OK;
}

int ensure_ng(rt_ctx* c)
{
    if (c->ng_out) return RT_OK;
    for (auto& p : c->ng_old) CK(dalloc(p, (size_t)c->g.N));
    CK(dalloc(c->ng_part, (size_t)ng_partial_size()));
    CK(dalloc(c->ng_out, 5));
    return RT_OK;
}

// Ng bookkeeping of iteration `it` (1-based), before its operator splitting
// produces J_new in c->Jn from c->J: c->J is remembered (hist: where the
// kernel that forms the outer delta copies it), and the iteration
// extrapolates (due) when four iterates are held and it is a multiple of the
// period.  Otherwise the operator-splitting kernel may form the delta itself.
int ng_begin(rt_ctx* c, int it, double* delta, double*& hist, bool& due)
{
    hist = nullptr;
    due = false;
    c->os_delta = c->os_hist = nullptr;
    if (!c->ng_period) {
        c->os_delta = delta;
        return RT_OK;
    }
    int rc = ensure_ng(c);
    if (rc) return rc;
    double* t = c->ng_old[2];
    c->ng_old[2] = c->ng_old[1];
    c->ng_old[1] = c->ng_old[0];
    c->ng_old[0] = hist = t;
    if (c->ng_count < 4) ++c->ng_count;
    due = c->ng_count == 4 && it % c->ng_period == 0 &&
          (it == 1 || c->ng_last_delta >= c->ng_min_delta);
    c->os_delta = due ? nullptr : delta;
    c->os_hist = due ? nullptr : hist;
    return RT_OK;
}

// After the operator splitting (in one kernel: one): where the extrapolation is
// due, the weighted sums and the extrapolation of J_new, whose 2x2 system is
// solved on the device (no host synchronisation; the iterate is left unchanged
// if it is singular); then the outer delta, unless that kernel has formed it.
int ng_end(rt_ctx* c, bool one, bool due, double* delta, double* hist)
{
    const bool formed = one && c->os_delta;
    c->os_delta = c->os_hist = nullptr;
    if (due) {
        CK(launch_ng_dots(c->g.N, c->Jn, c->J, c->ng_old[1], c->ng_old[2], c->ng_part,
                          c->ng_out, c->stream));
        CK(launch_ng_apply(c->g.N, c->ng_out, c->J, c->ng_old[1], c->Jn, c->stream));
        c->stats.launches += 3;
        c->ng_applied += 1;
        c->ng_count = 1;
    }
    if (!formed) {
        CK(launch_rel_change(c->g.N, c->Jn, c->J, delta, hist, c->stream));
        c->stats.launches += 1;
    }
    return RT_OK;
}

// After an iteration that failed: no history, no delta in the next solve.
void ng_forget(rt_ctx* c)
{
    c->ng_count = 1;
    c->os_delta = c->os_hist = nullptr;
}

// Switch between the FP32 sweep and the double-float march (see rt_set_precision).
int switch_precision(rt_ctx* c, int precision)
{
    if (precision == c->precision) return RT_OK;
    const bool ok = (precision == RT_FP32_SWEEP || precision == RT_DF64) &&
                    (c->precision == RT_FP32_SWEEP || c->precision == RT_DF64);
    if (!ok) return fail(c, RT_EINVAL, "precision switches only between RT_FP32_SWEEP and RT_DF64");
    if (precision == RT_FP32_SWEEP && c->fs_method == RT_FS_SHORT)
        return fail(c, RT_EINVAL, "short characteristics have no FP32-sweep form");
    int rc = form_buffers(c, precision);
    if (rc) return rc;
    c->precision = precision;
    c->rec_valid = false;
    c->gdiff_valid = false;    // the gradient's packed copy differs between the forms
    c->lstar_valid = c->coef_valid = false;   // Lambda* is rebuilt by the new form's kernel
    c->ng_count = 1;           // restart the Ng history with iterates of the new form
    return RT_OK;
}

int solve(rt_ctx* c, double tol, int max_iter, double tol_inner, int max_sweeps, double* J_out,
          int* iters, double* last_delta, double* deltas, int* sweeps, bool device)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((rc = need_all(c))) return rc;
    if (max_iter < 1 || max_sweeps < 1 || !(tol >= 0) || !(tol_inner >= 0))
        return fail(c, RT_EINVAL, "bad iteration controls");
    // finishing stage: the context leaves it, and gets its Ng threshold
    // back, when the solve ends, whichever way it ends
    struct FinishGuard {
        rt_ctx* c;
        double ng_min;
        bool on;
        ~FinishGuard()
        {
            if (on) {
                c->fin = 0;
                c->ng_min_delta = ng_min;
            }
        }
    } guard{c, c->ng_min_delta, false};
    int it = 0;
    double delta = 0.0;
    bool converged = false;
    unsigned long long total_steps = 0;
    while (it < max_iter) {
        if ((rc = prepare_source(c, nullptr, true, false))) return rc;
        if ((rc = run_fs(c, c->Jfs, true))) return rc;
        int ns = 0;
        double* hist = nullptr;
        bool due = false;
        if ((rc = ng_begin(c, it + 1, c->scal + 2, hist, due))) return rc;
        if ((rc = run_os(c, c->Jfs, c->J, c->Jn, tol_inner, max_sweeps, true, &ns))) {
            ng_forget(c);
            return rc;
        }
        if (!c->os_one) CK(cudaMemsetAsync(c->scal + 2, 0, sizeof(double), c->stream));
        if ((rc = ng_end(c, c->os_one, due, c->scal + 2, hist))) return rc;
        // with the sweep count where the step ran as one kernel
        CK(cudaMemcpyAsync(c->h_scal + 2, c->scal + 2, sizeof(double) * (c->os_one ? 3 : 1),
                           cudaMemcpyDeviceToHost, c->stream));
        CK(cudaStreamSynchronize(c->stream));
        c->stats.host_syncs += 1;
        c->stats.iterations += 1;
        harvest(c);
        if (ns < 0 && (rc = os_graph_done(c, &ns))) {
            ng_forget(c);       // its history may not have been written
            return rc;
        }
        total_steps += *c->h_steps;
        delta = c->h_scal[2];
        c->ng_last_delta = delta;
        double* t = c->J;
        c->J = c->Jn;
        c->Jn = t;
        if (deltas) deltas[it] = delta;
        if (sweeps) sweeps[it] = ns;
        ++it;
        if (tol > 0 && delta < tol) {
            converged = true;
            break;
        }
        if (!guard.on && c->df_switch > 0 && c->precision == RT_FP32_SWEEP && delta < c->df_switch) {
            c->fin = 1;               // next formal solution: the double-float reference
            c->ng_min_delta = 0.0;    // Ng on every period from here
            c->ng_count = 1;          // its history restarts with FP64-accurate iterates
            guard.on = true;
        }
    }
    c->last_steps = total_steps;
    c->stats.steps += total_steps;
    if (J_out) {
        CK(cudaMemcpyAsync(J_out, c->J, sizeof(double) * c->g.N,
                           device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, c->stream));
        CK(cudaStreamSynchronize(c->stream));
    }
    if (iters) *iters = it;
    if (last_delta) *last_delta = delta;
    if (tol > 0 && !converged)
        return fail(c, RT_ENOTCONV, "not converged after %d iterations (delta %.3e >= tol %.3e)",
                    it, delta, tol);
    return RT_OK;
}

// ---- batched wavelengths ----------------------------------------------------

}  // namespace

struct rt_batch {
    int device = 0;
    int precision = RT_FP32_SWEEP;
    cudaStream_t own_stream = nullptr;
    cudaStream_t stream = nullptr;
    int num_sms = 0;
    std::vector<rt_ctx*> ctx;       // one per wavelength, all on `stream`
    std::vector<int> order;         // problems by decreasing size (fused launch order)
    std::vector<int> iters;         // outer iterations done since the last reset
    std::vector<double> delta;      // last outer delta
    std::vector<char> converged;
    View32* d_views = nullptr;      // device copies of the per-problem FP32 views
    View32* h_views = nullptr;      // pinned host copies (uploaded when a view changes)
    std::vector<char> view_fin;     // problems whose device view is the finishing-stage one
    int* d_ids = nullptr;
    long long* d_prefix = nullptr;
    int* h_ids = nullptr;           // pinned
    long long* h_prefix = nullptr;  // pinned
    double* d_delta = nullptr;      // outer deltas [nprob]
    double* h_delta = nullptr;      // pinned
    unsigned long long* d_steps = nullptr;
    unsigned long long* h_steps = nullptr;
    int groups_req = 0;
    int threads32 = 0;              // threads per block of the fused FP32 launch (0: 128)
    bool profiling = false;
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
    bool jac_pending = false;
    // The operator-splitting step of all active problems as one CUDA graph:
    // per problem an independent branch (right-hand side, a device-side
    // WHILE loop of sweeps, the pick of the last sweep's buffer).  Keyed by
    // the active set and the buffers it touches; two cached instances,
    // because J and J_new alternate between two buffers.
    struct OsGraph {
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        std::vector<const void*> key;
    } osg[2];
    int osg_next = 0;
    bool use_graphs = true;
    // the active problems' solves in one kernel (launch_os_solve), where their
    // blocks are resident together: tasks and first blocks (device, pinned
    // copies), barrier words of all problems
    OsTask *d_tasks = nullptr, *h_tasks = nullptr;
    int *d_first = nullptr, *h_first = nullptr;
    unsigned long long* d_bdlt = nullptr;
    int bdlt_cap = 0;               // words per problem it holds
    bool os_one = false;            // the last step ran that way
    int* d_sweeps = nullptr;        // sweeps of each problem's last OS step
    int* h_sweeps = nullptr;        // pinned
    // Recorded marches: a problem starts iterating once its recording fits
    // in the batch's budget (rec_mode: -1 automatic, 0 off, > 0 bytes), so
    // that every problem records in its first formal solution as a single
    // solve does; its memory returns when it converges.
    long long rec_mode = -1;
    std::vector<char> admitted;
    // recording blocks returned by converged problems, handed to the next
    // admitted ones (a large cudaMalloc/cudaFree per problem costs tens of
    // milliseconds); freed when a solve ends
    std::vector<std::pair<char*, long long>> rec_pool;
    Rep32* d_rviews = nullptr;      // replay views (device) and pinned host copies
    Rep32* h_rviews = nullptr;
    int* d_rids = nullptr;
    long long* d_rprefix = nullptr;
    int* h_rids = nullptr;          // pinned
    long long* h_rprefix = nullptr; // pinned
    rt_stats stats{};
    std::string err;
};

namespace {

int bfail(rt_batch* b, int code, const char* fmt, ...)
{
    if (b) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof buf, fmt, ap);
        va_end(ap);
        b->err = buf;
    }
    return code;
}

#define BCK(call)                                                                       \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return bfail(b, e_ == cudaErrorMemoryAllocation ? RT_ENOMEM : RT_ECUDA,     \
                         "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
    } while (0)

// Propagate a per-problem failure with the problem's message.
int bpass(rt_batch* b, int p, int rc)
{
    if (rc == RT_OK) return RT_OK;
    return bfail(b, rc, "problem %d: %s", p, b->ctx[p]->err.c_str());
}

int batch_groups(const rt_batch* b, const std::vector<int>& act)
{
    if (b->groups_req > 0) return b->groups_req < kSlots ? b->groups_req : kSlots;
    long long blocks = 0;
    for (int p : act) blocks += fs32_blocks(b->ctx[p]->g, 1, b->threads32);
    int G = 1;
    while (G < kSlots && blocks * G < 64LL * (b->num_sms > 0 ? b->num_sms : 152)) G *= 2;
    return G;
}

// Free pooled blocks until at most `keep` bytes are held, the largest first;
// not block `pick`.
void batch_free_pool(rt_batch* b, long long keep = 0, char* pick = nullptr)
{
    long long held = 0;
    for (auto& blk : b->rec_pool) held += blk.second;
    if (held <= keep) return;
    cudaStreamSynchronize(b->stream);
    std::sort(b->rec_pool.begin(), b->rec_pool.end(),
              [](const auto& x, const auto& y) { return x.second < y.second; });
    for (size_t i = b->rec_pool.size(); i-- > 0 && held > keep;) {
        if (b->rec_pool[i].first == pick) continue;
        held -= b->rec_pool[i].second;
        cudaFree(b->rec_pool[i].first);
        b->rec_pool.erase(b->rec_pool.begin() + i);
    }
}

// What the batch's recordings may take: `used` of `limit` bytes are held or
// promised to the admitted problems that have not recorded yet; automatic:
// `reserve` of the `free_now` bytes of the device (less what is promised) stay free.
struct RecBudget {
    long long limit = 0, used = 0, reserve = 0, free_now = 0;
    bool automatic = false;
};

// Give problem c up to `want` bytes for its recording, with a pooled block to
// start from, where the budget has them; blocks it cannot use go back to the
// device where that makes the room.  op: what it will take is known when it
// records (ensure_op_rec), at most `want`; else it takes them now.
bool batch_take(rt_batch* b, rt_ctx* c, long long want, bool op, RecBudget& m)
{
    // the smallest block that holds it; for an operator else the largest
    int pick = -1;
    long long pooled = 0;
    for (size_t i = 0; i < b->rec_pool.size(); ++i) {
        const long long cap = b->rec_pool[i].second, best = pick < 0 ? 0 : b->rec_pool[pick].second;
        pooled += cap;
        if (cap >= want ? best < want || cap < best : op && cap > best) pick = (int)i;
    }
    char* mem = pick < 0 ? nullptr : b->rec_pool[pick].first;
    long long cap = pick < 0 ? 0 : b->rec_pool[pick].second;
    const long long work = op && !c->ow_mem ? op_work_bytes(c) : 0;
    auto room = [&](long long have, long long freed) {
        const long long grow = std::max(want - have, 0LL);
        return m.used + grow <= m.limit + freed &&
               (!m.automatic || grow + work == 0 || grow + work + m.reserve <= m.free_now + freed);
    };
    if (!room(cap, 0)) {
        if (!room(cap, pooled - cap)) {
            if (!room(0, pooled)) return false;
            mem = nullptr;
            cap = 0;
        }
        batch_free_pool(b, cap, mem);
        m.used -= pooled - cap;
        m.free_now += pooled - cap;
    }
    for (size_t i = 0; mem && i < b->rec_pool.size(); ++i)
        if (b->rec_pool[i].first == mem) {
            b->rec_pool.erase(b->rec_pool.begin() + i);
            c->rec_mem = mem;
            c->rec_cap = cap;
            break;
        }
    c->rec_mode = std::max(want, cap);
    if (!op) {
        bool use = false;
        if (ensure_rec(c, use) != RT_OK || !use) return false;
    }
    m.used += std::max(want - cap, 0LL);
    m.free_now -= std::max(want - cap, 0LL) + work;
    return true;
}

// Admit waiting problems (in launch order) whose recorded march fits in the
// batch's budget beside the recordings held; a problem whose form does not
// record, or whose recording could never fit, starts at once and marches.
// When nothing runs and a problem cannot get its memory, it starts marching
// too, so that the solve always progresses.
int batch_admit(rt_batch* b, int max_iter)
{
    RecBudget m;
    m.limit = b->rec_mode;
    m.automatic = b->rec_mode < 0;
    bool running = false;
    for (auto& blk : b->rec_pool) m.used += blk.second;
    if (m.automatic) {
        // automatic: recordings up to 60% of the device, each admitted only
        // while what the unconverged problems still allocate (Ng's iterates;
        // node lists; at their finishing stage the reference's double-float
        // node planes and tables, S_ref, J_ref and the source change) stays
        // free beside it, with 4 GiB to spare
        size_t fr = 0, tot = 0;
        BCK(cudaMemGetInfo(&fr, &tot));
        m.limit = (long long)(0.6 * (double)tot);
        m.free_now = (long long)fr;
        m.reserve = 4LL << 30;
    }
    for (size_t p = 0; p < b->ctx.size(); ++p) {
        const rt_ctx* c = b->ctx[p];
        const bool op = c->precision != RT_FP32_SWEEP;
        if (m.automatic && !b->converged[p] && !c->S_ref)
            m.reserve += 24 * c->g.N + (c->node4 ? 0 : 64 * c->g.N) +
                         (c->ng_old[0] ? 0 : 24 * c->g.N) +     // Ng's older iterates
                         36LL * c->g.ndir * c->g.nz + (1LL << 20);
        if (m.automatic && !b->converged[p] && op && !c->ol_mem && op_fits(c))
            m.reserve += op_list_bytes(c);
        m.used += c->rec_cap;
        if (!b->admitted[p] || b->converged[p] || b->iters[p] >= max_iter) continue;
        running = true;
        if (c->rec_valid || c->rec_mode <= c->rec_cap) continue;
        m.used += c->rec_mode - c->rec_cap;         // promised
        m.free_now -= c->rec_mode - c->rec_cap + (op && !c->ow_mem ? op_work_bytes(c) : 0);
    }
    for (int p : b->order) {
        rt_ctx* c = b->ctx[p];
        if (b->admitted[p] || b->converged[p] || b->iters[p] >= max_iter) continue;
        const bool op = c->precision != RT_FP32_SWEEP;
        const long long need = rec_need(c);
        if (b->rec_mode == 0 || need == 0 || need > m.limit) {
            c->rec_mode = 0;                      // marches
        } else {
            // room for the assembled operator where the budget allows it at
            // all, else (or where nothing runs whose memory could be waited for)
            // for the ray-by-ray recording
            const long long ask = op && rec_ask(c, need) <= m.limit ? rec_ask(c, need) : need;
            if (!batch_take(b, c, ask, op, m)) {
                if (running) continue;            // wait for memory
                if (ask == need || !batch_take(b, c, need, op, m)) c->rec_mode = 0;
            }
        }
        b->admitted[p] = 1;
        running = true;
    }
    return RT_OK;
}

// A problem that stops iterating returns its recording's memory to the
// batch's pool.
void batch_release(rt_batch* b, int p)
{
    rt_ctx* c = b->ctx[p];
    if (c->rec_cap) {
        cudaStreamSynchronize(b->stream);
        b->rec_pool.emplace_back(c->rec_mem, c->rec_cap);
        c->rec_mem = nullptr;
        c->rec_cap = 0;
        c->rec = FsRec{};
        c->rec32 = Rec32{};
        c->op = OpMap{};
        c->rec_op = false;
        c->srec = nullptr;
        c->rec_valid = false;
    }
    if (c->ow_mem) {
        cudaStreamSynchronize(b->stream);
        free_op_work(c);
    }
}

// What a batch keeps of its recordings' memory between solves (the blocks of
// a small batch: allocating and freeing 4 GB of them took 4 of 37 ms per solve
// of six wavelengths of 41^3 and 20^3); freed with the batch.
constexpr long long kPoolKeep = 8LL << 30;

void bharvest(rt_batch* b)
{
    float ms = 0.f;
    if (b->profiling && cudaEventElapsedTime(&ms, b->ev[0], b->ev[1]) == cudaSuccess)
        b->stats.fs_ms += ms;
    if (b->jac_pending && cudaEventElapsedTime(&ms, b->ev[2], b->ev[3]) == cudaSuccess)
        b->stats.jacobi_ms += ms;
    b->jac_pending = false;
}

void free_batch_graphs(rt_batch* b)
{
    for (auto& e : b->osg) {
        if (e.exec) cudaGraphExecDestroy(e.exec);
        if (e.graph) cudaGraphDestroy(e.graph);
        e = rt_batch::OsGraph{};
    }
}

std::vector<const void*> batch_graph_key(const rt_batch* b, const std::vector<int>& act,
                                         double tol, int max_sweeps)
{
    std::vector<const void*> k;
    k.push_back(reinterpret_cast<const void*>((intptr_t)max_sweeps));
    long long tb;
    std::memcpy(&tb, &tol, sizeof tb);
    k.push_back(reinterpret_cast<const void*>((intptr_t)tb));
    for (int p : act) {
        const rt_ctx* c = b->ctx[p];
        k.push_back(reinterpret_cast<const void*>((intptr_t)p));
        k.push_back(reinterpret_cast<const void*>((intptr_t)c->os_method));
        for (const void* q : {(const void*)c->J, (const void*)c->Jn, (const void*)c->Jfs,
                              (const void*)c->coef, (const void*)c->rdiag, (const void*)c->r,
                              (const void*)c->Ja, (const void*)c->Jb, (const void*)c->dlt,
                              (const void*)c->d_nsw})
            k.push_back(q);
    }
    return k;
}

// Capture the per-problem branches of the batch operator-splitting graph.
// Every capture that begins is ended, also after an error.
cudaError_t build_batch_os_graph(rt_batch* b, const std::vector<int>& act, double tol,
                                 int max_sweeps, cudaGraph_t* out)
{
    cudaGraph_t g = nullptr;
    cudaError_t err = cudaGraphCreate(&g, 0);
    if (err != cudaSuccess) return err;
    const cudaStream_t st = b->stream;
    for (int p : act) {
        rt_ctx* c = b->ctx[p];
        const bool gs = c->os_method == RT_OS_GAUSS_SEIDEL;
        cudaGraphConditionalHandle h;
        err = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault);
        if (err != cudaSuccess) break;
        // prologue, a branch of its own (no dependencies)
        err = cudaStreamBeginCaptureToGraph(st, g, nullptr, nullptr, 0,
                                            cudaStreamCaptureModeThreadLocal);
        if (err != cudaSuccess) break;
        std::vector<cudaGraphNode_t> deps;
        {
            cudaError_t e1 = launch_os_rhs(c->g, c->coef, c->rdiag, c->Jfs, c->J, c->r, gs, st);
            cudaError_t e2 = cudaMemsetAsync(c->dlt, 0, sizeof(double) * ((size_t)max_sweeps + kPassSweeps), st);
            cudaError_t e3 = cudaMemcpyAsync(c->Jb, c->J, sizeof(double) * c->g.N,
                                             cudaMemcpyDeviceToDevice, st);
            cudaError_t e4 = cudaMemsetAsync(c->d_nsw, 0, sizeof(int), st);
            cudaStreamCaptureStatus cs;
            const cudaGraphNode_t* dp = nullptr;
            size_t nd = 0;
            cudaError_t e5 = cudaStreamGetCaptureInfo(st, &cs, nullptr, nullptr, &dp, nullptr, &nd);
            if (e5 == cudaSuccess) deps.assign(dp, dp + nd);
            cudaGraph_t o = nullptr;
            cudaError_t e6 = cudaStreamEndCapture(st, &o);
            for (cudaError_t x : {e1, e2, e3, e4, e5, e6})
                if (err == cudaSuccess && x != cudaSuccess) err = x;
        }
        if (err != cudaSuccess) break;
        // the sweep loop
        cudaGraphNodeParams cp = {};
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        cudaGraphNode_t cn;
        err = cudaGraphAddNode(&cn, g, deps.data(), nullptr, deps.size(), &cp);
        if (err != cudaSuccess) break;
        err = cudaStreamBeginCaptureToGraph(st, cp.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                            cudaStreamCaptureModeThreadLocal);
        if (err != cudaSuccess) break;
        {
            cudaError_t e1 = launch_sweep_pass(c->g, c->coef, c->r, c->Ja, c->Jb, c->dlt, c->d_nsw,
                                               max_sweeps, tol, gs, h, st);
            cudaGraph_t o = nullptr;
            cudaError_t e2 = cudaStreamEndCapture(st, &o);
            err = e1 != cudaSuccess ? e1 : e2;
        }
        if (err != cudaSuccess) break;
        // epilogue: the last sweep's iterate into J_new, after the loop
        err = cudaStreamBeginCaptureToGraph(st, g, &cn, nullptr, 1, cudaStreamCaptureModeThreadLocal);
        if (err != cudaSuccess) break;
        {
            cudaError_t e1 = launch_os_select(c->g.N, c->dlt, max_sweeps, tol, c->Ja, c->Jb, c->Jn,
                                              b->d_sweeps + p, st);
            cudaGraph_t o = nullptr;
            cudaError_t e2 = cudaStreamEndCapture(st, &o);
            err = e1 != cudaSuccess ? e1 : e2;
        }
        if (err != cudaSuccess) break;
    }
    if (err != cudaSuccess) {
        cudaGraphDestroy(g);
        return err;
    }
    *out = g;
    return cudaSuccess;
}

// Formal solutions of the active problems: FP32 sweep in one fused launch,
// FP64 one launch per problem.
int batch_fs(rt_batch* b, const std::vector<int>& act)
{
    int rc;
    std::vector<char> direct(b->ctx.size(), 0);     // J is in c->Jfs already
    for (int p : act) {
        rt_ctx* c = b->ctx[p];
        if ((rc = bpass(b, p, prepare_source(c, nullptr, true, false)))) return rc;
        if ((rc = bpass(b, p, fs_prepare(c)))) return rc;
    }
    const int G = batch_groups(b, act);
    BCK(cudaMemsetAsync(b->d_steps, 0, sizeof(unsigned long long), b->stream));
    if (b->profiling) BCK(cudaEventRecord(b->ev[0], b->stream));
    if (b->precision == RT_FP32_SWEEP) {
        // problems holding a recording: record it in their first formal
        // solution, then one fused replay over all of them (their source, or
        // in the finishing stage its change, packed for the replay)
        long long rtotal = 0;
        int rq = 0;
        std::vector<char> replays(b->ctx.size(), 0);
        for (int p : act) {
            rt_ctx* c = b->ctx[p];
            if (c->precision != RT_FP32_SWEEP || c->fin == 1) continue;
            bool use = false;
            if ((rc = bpass(b, p, ensure_rec(c, use)))) return rc;
            if (!use) continue;
            if (!c->rec_valid) {
                if (c->fin != 0) continue;
                BCK(launch_fs32rec(view32(c), cut_of(c) * kRecCutMargin, G, c->rec32, b->d_steps,
                                   b->stream));
                c->rec_valid = true;
                b->stats.launches += 1;
            }
            if ((rc = bpass(b, p, rep_source(c)))) return rc;
            b->h_rviews[p] = Rep32{c->g, c->srec, c->info, c->poff32, c->bw32, c->rec32,
                                   c->partial, c->fin == 2 ? 1 : 0, plane_major32(c->g, c->order32)};
            b->h_rids[rq] = p;
            b->h_rprefix[rq] = rtotal;
            rtotal += fs32_blocks(c->g, G, b->threads32);
            ++rq;
            replays[p] = 1;
        }
        b->h_rprefix[rq] = rtotal;
        if (rq > 0) {
            BCK(cudaMemcpyAsync(b->d_rviews, b->h_rviews, sizeof(Rep32) * b->ctx.size(),
                                cudaMemcpyHostToDevice, b->stream));
            BCK(cudaMemcpyAsync(b->d_rids, b->h_rids, sizeof(int) * rq, cudaMemcpyHostToDevice,
                                b->stream));
            BCK(cudaMemcpyAsync(b->d_rprefix, b->h_rprefix, sizeof(long long) * (rq + 1),
                                cudaMemcpyHostToDevice, b->stream));
            BCK(launch_fs32rep_batch(b->d_rviews, b->d_rids, b->d_rprefix, rq, rtotal, G,
                                     b->threads32, b->d_steps, b->stream));
            b->stats.fs_launches += 1;
            b->stats.launches += 1;
        }
        // one fused launch over the other problems in the FP32 sweep, including
        // those marching their source change in the finishing stage (act is
        // in launch order); a finishing-stage reference and problems switched
        // to the double-float march by hand run one launch each
        long long total = 0;
        int q = 0;
        for (int p : act) {
            rt_ctx* c = b->ctx[p];
            if (c->precision != RT_FP32_SWEEP || c->fin == 1 || replays[p]) continue;
            const char want = c->fin == 2;
            if (b->view_fin[p] != want) {     // this problem's view changed form
                b->h_views[p] = want ? view32_fin(c) : view32(c);
                BCK(cudaMemcpyAsync(b->d_views + p, b->h_views + p, sizeof(View32),
                                    cudaMemcpyHostToDevice, b->stream));
                b->view_fin[p] = want;
            }
            b->h_ids[q] = p;
            b->h_prefix[q] = total;
            total += fs32_blocks(c->g, G, b->threads32);
            ++q;
        }
        b->h_prefix[q] = total;
        if (q > 0) {
            BCK(cudaMemcpyAsync(b->d_ids, b->h_ids, sizeof(int) * q, cudaMemcpyHostToDevice,
                                b->stream));
            BCK(cudaMemcpyAsync(b->d_prefix, b->h_prefix, sizeof(long long) * (q + 1),
                                cudaMemcpyHostToDevice, b->stream));
            BCK(launch_fs32_batch(b->d_views, b->d_ids, b->d_prefix, q, total, G, b->threads32,
                                  cut_of(b->ctx[0]), b->d_steps, b->stream));
            b->stats.fs_launches += 1;
            b->stats.launches += 1;
        }
        for (int p : act) {
            rt_ctx* c = b->ctx[p];
            if (c->precision == RT_DF64) {
                bool d = false;
                if ((rc = bpass(b, p, df_formal(c, G, c->Jfs, b->d_steps, d)))) return rc;
                direct[p] = d;
            } else if (c->fin == 1) {
                if ((rc = bpass(b, p, fin_reference_march(c, G, b->d_steps, b->stream)))) return rc;
            } else {
                continue;
            }
            b->stats.fs_launches += 1;
            b->stats.launches += 1;
        }
    } else {
        for (int p : act) {
            rt_ctx* c = b->ctx[p];
            bool d = false;
            rc = b->precision == RT_DF64 ? df_formal(c, G, c->Jfs, b->d_steps, d)
                                         : fs64_formal(c, G, c->Jfs, b->d_steps, d);
            if ((rc = bpass(b, p, rc))) return rc;
            direct[p] = d;
            if (!c->rec_valid && c->rec_mode != 0) {    // no memory: marches from here on
                batch_release(b, p);
                c->rec_mode = 0;
            }
            b->stats.fs_launches += 1;
            b->stats.launches += 1;
        }
    }
    if (b->profiling) BCK(cudaEventRecord(b->ev[1], b->stream));
    for (int p : act) {
        rt_ctx* c = b->ctx[p];
        if ((rc = bpass(b, p, fs_finish(c, c->Jfs, direct[p])))) return rc;
        if (c->precision == RT_FP32_SWEEP && c->fin == 1 &&
            (rc = bpass(b, p, fin_record(c, c->Jfs, b->stream))))
            return rc;
    }
    BCK(cudaMemcpyAsync(b->h_steps, b->d_steps, sizeof(unsigned long long), cudaMemcpyDeviceToHost,
                        b->stream));
    return RT_OK;
}

// Operator-splitting solves of the active problems in one cooperative kernel,
// where all their blocks are resident together; ran: whether it was launched.
int batch_os_one(rt_batch* b, const std::vector<int>& act, double tol_inner, int max_sweeps, bool& ran)
{
    ran = false;
    b->os_one = false;
    const int P = (int)b->ctx.size(), method = b->ctx[act[0]]->os_method;
    long long total = 0;
    for (int p : act) {
        if (b->ctx[p]->os_method != method) return RT_OK;
        total += b->ctx[p]->g.N;
    }
    OsShape sh;
    os_solve_shape(total, b->num_sms, method == RT_OS_GAUSS_SEIDEL, &sh);
    if (sh.blocks == 0 || P * os_barriers(b->ctx[act[0]], max_sweeps) > kBarWords) return RT_OK;
    if (!b->d_tasks) BCK(cudaMalloc((void**)&b->d_tasks, sizeof(OsTask) * P));
    if (!b->d_first) BCK(cudaMalloc((void**)&b->d_first, sizeof(int) * P));
    if (!b->h_tasks) BCK(cudaMallocHost((void**)&b->h_tasks, sizeof(OsTask) * P));
    if (!b->h_first) BCK(cudaMallocHost((void**)&b->h_first, sizeof(int) * P));
    const int words = (int)os_barriers(b->ctx[act[0]], max_sweeps);
    if (b->bdlt_cap < words) {
        dfree(b->d_bdlt);
        b->bdlt_cap = 0;
        BCK(cudaMalloc((void**)&b->d_bdlt, sizeof(unsigned long long) * (size_t)P * words));
        b->bdlt_cap = words;
    }
    const long long per = (long long)sh.threads * sh.voxels;
    sh.blocks = 0;
    for (size_t q = 0; q < act.size(); ++q) {
        rt_ctx* c = b->ctx[act[q]];
        const int nblk = (int)((c->g.N + per - 1) / per);
        b->h_tasks[q] = os_task(c, c->Jfs, c->J, c->Jn, b->d_bdlt + q * words,
                                b->d_sweeps + act[q], nblk);
        b->h_first[q] = sh.blocks;
        sh.blocks += nblk;
    }
    BCK(cudaMemcpyAsync(b->d_tasks, b->h_tasks, sizeof(OsTask) * act.size(), cudaMemcpyHostToDevice,
                        b->stream));
    BCK(cudaMemcpyAsync(b->d_first, b->h_first, sizeof(int) * act.size(), cudaMemcpyHostToDevice,
                        b->stream));
    BCK(cudaMemsetAsync(b->d_bdlt, 0, sizeof(unsigned long long) * act.size() * words, b->stream));
    if (b->profiling) BCK(cudaEventRecord(b->ev[2], b->stream));
    const cudaError_t e = launch_os_solve(b->h_tasks[0], b->d_tasks, b->d_first, (int)act.size(), sh,
                                          method == RT_OS_GAUSS_SEIDEL, b->num_sms, max_sweeps, tol_inner,
                                          b->stream);
    if (e == cudaErrorCooperativeLaunchTooLarge) return RT_OK;
    BCK(e);
    if (b->profiling) {
        BCK(cudaEventRecord(b->ev[3], b->stream));
        b->jac_pending = true;
    }
    b->os_one = ran = true;
    return RT_OK;
}

// Operator-splitting solves of the active problems as one kernel or one graph
// launch (no host synchronisation); the sweep counts reach b->d_sweeps.
int batch_os_graph(rt_batch* b, const std::vector<int>& act, double tol_inner, int max_sweeps)
{
    int rc;
    for (int p : act)
        if ((rc = bpass(b, p, ensure_coef(b->ctx[p])))) return rc;
    bool ran = false;
    if ((rc = batch_os_one(b, act, tol_inner, max_sweeps, ran)) || ran) return rc;
    for (int p : act) {
        rt_ctx* c = b->ctx[p];
        if ((rc = bpass(b, p, ensure_dlt(c, (long long)max_sweeps + kPassSweeps)))) return rc;
        if (!c->d_nsw) BCK(cudaMalloc((void**)&c->d_nsw, sizeof(int)));
    }
    std::vector<const void*> key = batch_graph_key(b, act, tol_inner, max_sweeps);
    rt_batch::OsGraph* e = nullptr;
    for (auto& x : b->osg)
        if (x.exec && x.key == key) e = &x;
    if (!e) {
        e = &b->osg[b->osg_next];
        b->osg_next ^= 1;
        if (e->exec) cudaGraphExecDestroy(e->exec);
        if (e->graph) cudaGraphDestroy(e->graph);
        *e = rt_batch::OsGraph{};
        cudaGraph_t g = nullptr;
        cudaError_t err = build_batch_os_graph(b, act, tol_inner, max_sweeps, &g);
        cudaGraphExec_t exec = nullptr;
        if (err == cudaSuccess) {
            err = cudaGraphInstantiate(&exec, g, 0);
            if (err != cudaSuccess) cudaGraphDestroy(g);
        }
        if (err != cudaSuccess) {
            cudaGetLastError();
            return bfail(b, RT_ECUDA, "building the batch operator-splitting graph: %s",
                         cudaGetErrorString(err));
        }
        e->graph = g;
        e->exec = exec;
        e->key.swap(key);
        b->stats.launches += 0;
    }
    if (b->profiling) BCK(cudaEventRecord(b->ev[2], b->stream));
    BCK(cudaGraphLaunch(e->exec, b->stream));
    if (b->profiling) {
        BCK(cudaEventRecord(b->ev[3], b->stream));
        b->jac_pending = true;
    }
    return RT_OK;
}

// Launch counts of the graph-driven operator splitting of `act`, from the
// sweep counts the graph wrote (read after the iteration's synchronisation).
int batch_os_graph_counts(rt_batch* b, const std::vector<int>& act)
{
    if (b->os_one) b->stats.launches += 1;
    for (int p : act) {
        if (b->h_sweeps[p] < 0)
            return bfail(b, RT_ETIMEOUT, "problem %d: a wait of the operator-splitting kernel gave up", p);
        const int per = b->ctx[p]->os_method == RT_OS_GAUSS_SEIDEL ? 2 : 1;
        const int passes = (b->h_sweeps[p] + kPassSweeps - 1) / kPassSweeps;
        b->stats.launches += b->os_one ? 0 : 2 + passes * (kPassSweeps * per + 1);
        b->stats.jacobi_launches += b->os_one ? b->h_sweeps[p] * per : passes * kPassSweeps * per;
    }
    return RT_OK;
}

// Operator-splitting solves of the active problems without graphs; sweeps
// are enqueued in chunks for every problem still iterating and checked with
// one host sync per chunk (a sweep after a converged one is a device-side
// no-op).
int batch_os(rt_batch* b, const std::vector<int>& act, double tol_inner, int max_sweeps)
{
    int rc;
    std::vector<int> inner;
    for (int p : act) {
        rt_ctx* c = b->ctx[p];
        if ((rc = bpass(b, p, ensure_coef(c)))) return rc;
        if ((rc = bpass(b, p, ensure_dlt(c, max_sweeps)))) return rc;
        BCK(launch_os_rhs(c->g, c->coef, c->rdiag, c->Jfs, c->J, c->r,
                          c->os_method == RT_OS_GAUSS_SEIDEL, b->stream));
        BCK(cudaMemsetAsync(c->dlt, 0, sizeof(double) * max_sweeps, b->stream));
        b->stats.launches += 1;
        inner.push_back(p);
    }
    std::vector<int> sweeps(b->ctx.size(), max_sweeps);
    int launched = 0, chunk = 2;
    while (!inner.empty() && launched < max_sweeps) {
        const int n0 = launched;
        const int n1 = launched + chunk < max_sweeps ? launched + chunk : max_sweeps;
        for (int p : inner) {
            rt_ctx* c = b->ctx[p];
            for (int n = n0; n < n1; ++n) {
                const double* cur = n == 0 ? c->J : (n & 1 ? c->Ja : c->Jb);
                double* nxt = n & 1 ? c->Jb : c->Ja;
                if (c->os_method == RT_OS_GAUSS_SEIDEL)
                    BCK(launch_gs_sweep(c->g, c->coef, c->r, cur, nxt, c->dlt, n, tol_inner,
                                        b->stream));
                else
                    BCK(launch_jacobi(c->g, c->coef, c->r, cur, nxt, c->dlt, n, tol_inner,
                                      b->stream));
            }
            BCK(cudaMemcpyAsync(c->h_dlt + n0, c->dlt + n0, sizeof(double) * (n1 - n0),
                                cudaMemcpyDeviceToHost, b->stream));
            const int per = c->os_method == RT_OS_GAUSS_SEIDEL ? 2 : 1;
            b->stats.launches += per * (n1 - n0);
            b->stats.jacobi_launches += per * (n1 - n0);
        }
        BCK(cudaStreamSynchronize(b->stream));
        b->stats.host_syncs += 1;
        std::vector<int> still;
        for (int p : inner) {
            rt_ctx* c = b->ctx[p];
            int done = -1;
            for (int n = n0; n < n1; ++n)
                if (c->h_dlt[n] < tol_inner) {
                    done = n;
                    break;
                }
            if (done >= 0) sweeps[p] = done + 1; else still.push_back(p);
        }
        inner.swap(still);
        launched = n1;
        if (chunk < 32) chunk *= 2;
    }
    for (int p : act) {
        rt_ctx* c = b->ctx[p];
        BCK(cudaMemcpyAsync(c->Jn, (sweeps[p] - 1) & 1 ? c->Jb : c->Ja, sizeof(double) * c->g.N,
                            cudaMemcpyDeviceToDevice, b->stream));
    }
    return RT_OK;
}

}  // namespace

extern "C" {

const char* rt_version(void) { return "rt3d 0.1 (sm_103a)"; }

int rt_create(rt_ctx** out, int device, int precision)
{
    if (!out) return RT_EINVAL;
    *out = nullptr;
    if (precision != RT_FP64 && precision != RT_FP32_SWEEP && precision != RT_DF64) return RT_EINVAL;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return RT_ECUDA;
    rt_ctx* c = new rt_ctx();
    c->device = device;
    c->precision = precision;
    if (cudaSetDevice(device) != cudaSuccess ||
        cudaStreamCreateWithFlags(&c->own_stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaMalloc((void**)&c->scal, 5 * sizeof(double)) != cudaSuccess ||
        cudaMalloc((void**)&c->d_steps, sizeof(unsigned long long)) != cudaSuccess ||
        cudaMallocHost((void**)&c->h_scal, 5 * sizeof(double)) != cudaSuccess ||
        cudaMallocHost((void**)&c->h_steps, sizeof(unsigned long long)) != cudaSuccess ||
        cudaEventCreate(&c->ev[0]) != cudaSuccess || cudaEventCreate(&c->ev[1]) != cudaSuccess ||
        cudaEventCreate(&c->ev[2]) != cudaSuccess || cudaEventCreate(&c->ev[3]) != cudaSuccess) {
        rt_destroy(c);
        return RT_ECUDA;
    }
    *c->h_steps = 0;
    c->d_sw = reinterpret_cast<int*>(c->scal + 4);
    c->h_sw = reinterpret_cast<int*>(c->h_scal + 4);
    c->stream = c->own_stream;
    // the FP32 sweep finishes in double-float by default (rt_set_df_finish)
    c->df_switch = precision == RT_FP32_SWEEP ? kDefaultDfSwitch : 0.0;
    c->g.top_bc = RT_BC_ZERO;
    c->g.bottom_bc = RT_BC_PLANCK;
#ifdef RT_CHECKED
    if (cudaMalloc((void**)&c->berr, 4 * sizeof(unsigned long long)) != cudaSuccess ||
        cudaMemset(c->berr, 0, 4 * sizeof(unsigned long long)) != cudaSuccess) {
        rt_destroy(c);
        return RT_ECUDA;
    }
#endif
    c->g.berr = c->berr;
    *out = c;
    return RT_OK;
}

int rt_destroy(rt_ctx* c)
{
    if (!c) return RT_OK;
    cudaSetDevice(c->device);
    if (c->stream) cudaStreamSynchronize(c->stream);
    free_grid_buffers(c);
    free_tables(c);
    dfree(c->scal);
    dfree(c->d_steps);
    dfree(c->berr);
    if (c->d_nsw) cudaFree(c->d_nsw);
    c->d_nsw = nullptr;
    dfree(c->os_words);
    if (c->h_scal) cudaFreeHost(c->h_scal);
    if (c->h_steps) cudaFreeHost(c->h_steps);
    if (c->h_dlt) cudaFreeHost(c->h_dlt);
    dfree(c->dlt);
    for (auto& e : c->ev)
        if (e) cudaEventDestroy(e);
    if (c->own_stream) cudaStreamDestroy(c->own_stream);
    delete c;
    return RT_OK;
}

const char* rt_last_error(const rt_ctx* c) { return c ? c->err.c_str() : "null context"; }

int rt_set_stream(rt_ctx* c, void* stream)
{
    int rc = enter(c);
    if (rc) return rc;
    CK(cudaStreamSynchronize(c->stream));
    c->stream = stream ? (cudaStream_t)stream : c->own_stream;
    return RT_OK;
}

int rt_set_grid(rt_ctx* c, int nx, int ny, int nz, double dx, double dy, double dz)
{
    int rc = enter(c);
    if (rc) return rc;
    if (nx < 3 || ny < 3 || nz < 2 || nz > 65535)
        return fail(c, RT_EINVAL, "grid %dx%dx%d: need nx, ny >= 3 and 2 <= nz <= 65535", nx, ny,
                    nz);
    if (!(dx > 0) || !(dy > 0) || !(dz > 0) || !std::isfinite(dx) || !std::isfinite(dy) ||
        !std::isfinite(dz))
        return fail(c, RT_EINVAL, "spacings must be finite and > 0");
    if ((long long)nx * ny > (1LL << 30) || (long long)nx * ny * nz > (1LL << 40))
        return fail(c, RT_EINVAL, "grid too large");
    if (c->precision != RT_FP64 && (2LL * ny + 1) * 2LL * nx * nz >= (1LL << 31))
        return fail(c, RT_EINVAL,
                    "grid too large for the FP32-sweep and double-float forms "
                    "((2ny+1)*2nx*nz >= 2^31)");
    CK(cudaStreamSynchronize(c->stream));
    free_grid_buffers(c);
    free_tables(c);
    c->have_grid = c->have_quad = c->have_chi = c->have_eps = c->have_B = false;
    c->lstar_valid = c->coef_valid = c->b2_valid = c->rec_valid = false;
    c->g.nx = nx; c->g.ny = ny; c->g.nz = nz;
    c->g.N = (long long)nx * ny * nz;
    c->g.ndir = 0;
    c->dx = dx; c->dy = dy; c->dz = dz;
    const size_t N = (size_t)c->g.N;
    CK(dalloc(c->chi, N)); CK(dalloc(c->eps, N)); CK(dalloc(c->B, N)); CK(dalloc(c->J, N));
    CK(dalloc(c->S, N)); CK(dalloc(c->Jfs, N)); CK(dalloc(c->Jn, N)); CK(dalloc(c->Ja, N));
    // r, 1/diag and c sized for either storage (colour-split >= N)
    const size_t Ns = (size_t)os_coef_stride(c->g, true);
    CK(dalloc(c->Jb, N)); CK(dalloc(c->r, Ns)); CK(dalloc(c->rdiag, Ns));
    CK(dalloc(c->lstar, 27 * N)); CK(dalloc(c->coef, 27 * Ns));
    CK(dalloc(c->gdiff, (size_t)nx * ny));
    CK(dalloc(c->zorder, (size_t)nz)); CK(dalloc(c->zscratch, 2 * (size_t)nz));
    if (c->precision != RT_FP64) {
        CK(dalloc(c->b2, (size_t)8 * nx * ny));
        CK(dalloc(c->g2, (size_t)4 * nx * ny));
    }
    c->have_grid = true;
    return form_buffers(c, c->precision);
}

int rt_set_boundary(rt_ctx* c, int top_mode, int bottom_mode)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((top_mode != RT_BC_ZERO && top_mode != RT_BC_PLANCK) ||
        (bottom_mode != RT_BC_ZERO && bottom_mode != RT_BC_PLANCK && bottom_mode != RT_BC_DIFFUSION))
        return fail(c, RT_EINVAL, "boundary modes: top ZERO or PLANCK, bottom ZERO, PLANCK or DIFFUSION");
    c->g.top_bc = top_mode;
    c->g.bottom_bc = bottom_mode;
    c->gdiff_valid = c->rec_valid = false;
    return RT_OK;
}

int rt_set_quadrature(rt_ctx* c, int ndir, const double* mu, const double* phi, const double* w)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((rc = need(c, c->have_grid, "the grid"))) return rc;
    if (ndir < 1 || !mu || !phi || !w) return fail(c, RT_EINVAL, "bad quadrature arrays");
    double sw = 0.0;
    for (int d = 0; d < ndir; ++d) {
        if (!std::isfinite(mu[d]) || !std::isfinite(phi[d]) || !std::isfinite(w[d]))
            return fail(c, RT_EINVAL, "direction %d is not finite", d);
        if (!(std::fabs(mu[d]) >= 1e-6) || !(std::fabs(mu[d]) <= 1.0))
            return fail(c, RT_EINVAL, "mu[%d] = %g: need 1e-6 <= |mu| <= 1", d, mu[d]);
        if (!(w[d] >= 0)) return fail(c, RT_EINVAL, "w[%d] = %g < 0", d, w[d]);
        sw += w[d];
    }
    if (std::fabs(sw - 1.0) > 1e-12) return fail(c, RT_EINVAL, "weights sum to %.17g, not 1", sw);
    CK(cudaStreamSynchronize(c->stream));
    free_tables(c);
    c->have_quad = false;
    c->g.ndir = ndir;
    const size_t T = (size_t)ndir * c->g.nz;
    CK(dalloc(c->d_mu, ndir)); CK(dalloc(c->d_phi, ndir)); CK(dalloc(c->d_w, ndir));
    CK(dalloc(c->info, ndir)); CK(dalloc(c->off, T)); CK(dalloc(c->bw, T));
    CK(dalloc(c->bwh, T)); CK(dalloc(c->bw32, T));
    CK(cudaMemcpyAsync(c->d_mu, mu, sizeof(double) * ndir, cudaMemcpyHostToDevice, c->stream));
    CK(cudaMemcpyAsync(c->d_phi, phi, sizeof(double) * ndir, cudaMemcpyHostToDevice, c->stream));
    CK(cudaMemcpyAsync(c->d_w, w, sizeof(double) * ndir, cudaMemcpyHostToDevice, c->stream));
    CK(launch_dir_tables(c->g, c->dx, c->dy, c->dz, c->d_mu, c->d_phi, c->d_w, c->info, c->off,
                         c->bw, c->bwh, c->bw32, c->stream));
    c->stats.launches += 1;
    if (c->precision != RT_FP64) {
        CK(dalloc(c->poff, T));
        CK(dalloc(c->poff32, T));
        CK(launch_pad_offsets(c->g, c->info, c->off, 2LL * c->g.ny, c->poff, c->stream));
        CK(launch_pad_offsets(c->g, c->info, c->off, 2LL * c->g.ny + 1, c->poff32, c->stream));
        c->stats.launches += 2;
    } else {
        CK(dalloc(c->dn, (size_t)ndir));
        CK(launch_down_tables(c->g, c->dx, c->dy, c->dz, c->d_mu, c->d_phi, c->dn, c->stream));
        c->stats.launches += 1;
    }
    c->wsum = sw;
    c->dord.resize(ndir);
    for (int d = 0; d < ndir; ++d) c->dord[d] = d;
    std::stable_sort(c->dord.begin(), c->dord.end(), [mu](int a, int b) {
        if ((mu[a] > 0) != (mu[b] > 0)) return mu[a] > 0;
        return std::fabs(mu[a]) > std::fabs(mu[b]);
    });
    c->dpos = 0;
    for (int d = 0; d < ndir; ++d) c->dpos += mu[d] > 0;
    c->have_quad = true;
    if ((rc = form_buffers(c, c->precision))) {
        c->have_quad = false;
        return rc;
    }
    CK(cudaStreamSynchronize(c->stream));
    c->lstar_valid = c->coef_valid = c->rec_valid = false;
    return RT_OK;
}

static int set_chi(rt_ctx* c, const double* chi, bool device)
{
    int rc = set_field(c, chi, c ? c->chi : nullptr, device, "chi", true, false);
    if (rc) return rc;
    // the planes' dispatch order follows the new opacities (stream-ordered
    // before any march that reads it)
    CK(launch_plane_order(c->g, c->dz, c->chi, c->zscratch, c->zorder, c->stream));
    c->g.zorder = c->zorder;
    c->stats.launches += c->g.nz <= kRankOne ? 2 : 3;
    c->have_chi = true;
    c->lstar_valid = c->coef_valid = c->gdiff_valid = c->rec_valid = false;
    return RT_OK;
}

static int set_eps(rt_ctx* c, const double* eps, bool device)
{
    int rc = set_field(c, eps, c ? c->eps : nullptr, device, "eps", false, true);
    if (rc) return rc;
    c->have_eps = true;
    c->coef_valid = false;
    return RT_OK;
}

static int set_B(rt_ctx* c, const double* B, bool device)
{
    int rc = set_field(c, B, c ? c->B : nullptr, device, "B", false, false);
    if (rc) return rc;
    CK(cudaMemcpyAsync(c->J, c->B, sizeof(double) * c->g.N, cudaMemcpyDeviceToDevice, c->stream));
    c->ng_count = 1;
    c->ng_last_delta = 0.0;
    c->have_B = true;
    c->b2_valid = c->gdiff_valid = c->rec_valid = false;
    return RT_OK;
}

int rt_set_opacity(rt_ctx* c, const double* chi) { return set_chi(c, chi, false); }
int rt_set_epsilon(rt_ctx* c, const double* eps) { return set_eps(c, eps, false); }
int rt_set_planck(rt_ctx* c, const double* B) { return set_B(c, B, false); }
int rt_set_opacity_dev(rt_ctx* c, const double* chi) { return set_chi(c, chi, true); }
int rt_set_epsilon_dev(rt_ctx* c, const double* eps) { return set_eps(c, eps, true); }
int rt_set_planck_dev(rt_ctx* c, const double* B) { return set_B(c, B, true); }

int rt_formal_solution(rt_ctx* c, const double* S, double* J_fs, double* lstar)
{
    return check_bounds(c, formal_solution(c, S, J_fs, lstar, false));
}

int rt_formal_solution_dev(rt_ctx* c, const double* S, double* J_fs, double* lstar)
{
    return check_bounds(c, formal_solution(c, S, J_fs, lstar, true));
}

int rt_os_step(rt_ctx* c, const double* J_fs, const double* J_old, double* J_new, double tol_inner,
               int max_sweeps, int* sweeps)
{
    return check_bounds(c, os_step(c, J_fs, J_old, J_new, tol_inner, max_sweeps, sweeps, false));
}

int rt_os_step_dev(rt_ctx* c, const double* J_fs, const double* J_old, double* J_new,
                   double tol_inner, int max_sweeps, int* sweeps)
{
    return check_bounds(c, os_step(c, J_fs, J_old, J_new, tol_inner, max_sweeps, sweeps, true));
}

int rt_solve(rt_ctx* c, double tol, int max_iter, double tol_inner, int max_sweeps, double* J_out,
             int* iters, double* last_delta, double* deltas, int* sweeps)
{
    return check_bounds(c, solve(c, tol, max_iter, tol_inner, max_sweeps, J_out, iters, last_delta,
                                 deltas, sweeps, false));
}

int rt_solve_dev(rt_ctx* c, double tol, int max_iter, double tol_inner, int max_sweeps,
                 double* J_out, int* iters, double* last_delta, double* deltas, int* sweeps)
{
    return check_bounds(c, solve(c, tol, max_iter, tol_inner, max_sweeps, J_out, iters, last_delta,
                                 deltas, sweeps, true));
}

int rt_get_J(rt_ctx* c, double* J)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((rc = need(c, c->have_B, "the Planck function (initial J)"))) return rc;
    if (!J) return fail(c, RT_EINVAL, "J is NULL");
    CK(cudaMemcpyAsync(J, c->J, sizeof(double) * c->g.N, cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    return RT_OK;
}

int rt_set_J(rt_ctx* c, const double* J)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((rc = need(c, c->have_B, "the Planck function"))) return rc;
    if (!J) return fail(c, RT_EINVAL, "J is NULL");
    if ((rc = check_field(c, J, "J", false, false))) return rc;
    CK(cudaMemcpyAsync(c->J, J, sizeof(double) * c->g.N, cudaMemcpyHostToDevice, c->stream));
    c->ng_count = 1;
    CK(cudaStreamSynchronize(c->stream));
    return RT_OK;
}

// Diagnostics: one FP32 march of the source S (host, or NULL for
// eps B + (1 - eps) J) through the branch-counting kernel instantiation.
static int fs32_branch_counts(rt_ctx* c, const double* S, unsigned long long* steps,
                              unsigned long long* series)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((rc = need_all(c))) return rc;
    if (!steps || !series) return fail(c, RT_EINVAL, "steps or series is NULL");
    if (c->precision != RT_FP32_SWEEP || c->fs_method != RT_FS_LONG)
        return fail(c, RT_EINVAL, "branch counts need the FP32-sweep long-characteristics march");
    if ((rc = prepare_source(c, S, false, true))) return rc;
    if ((rc = fs_prepare(c))) return rc;
    CK(launch_pack_pairs(c->g, c->chi, c->S, c->pair, c->plo, c->stream));
    unsigned long long* d = nullptr;
    CK(cudaMalloc((void**)&d, 2 * sizeof(unsigned long long)));
    unsigned long long h[2] = {0, 0};
    cudaError_t e = cudaMemsetAsync(d, 0, 2 * sizeof(unsigned long long), c->stream);
    if (e == cudaSuccess)
        e = launch_fs32d(view32(c), cut_of(c), auto_groups(c), c->threads32, d, c->stream, d + 1);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(h, d, sizeof h, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    cudaFree(d);
    if (e != cudaSuccess) return fail(c, RT_ECUDA, "CUDA error %s", cudaGetErrorString(e));
    c->stats.launches += 1;
    *steps = h[0];
    *series = h[1];
    return RT_OK;
}

int rt_fs32_branch_counts(rt_ctx* c, const double* S, unsigned long long* steps,
                          unsigned long long* series)
{
    return check_bounds(c, fs32_branch_counts(c, S, steps, series));
}

int rt_last_step_count(rt_ctx* c, unsigned long long* steps)
{
    if (!c || !steps) return RT_EINVAL;
    *steps = c->last_steps;
    return RT_OK;
}

int rt_set_direction_groups(rt_ctx* c, int groups)
{
    if (!c) return RT_EINVAL;
    if (groups < 0 || groups > kSlots) return fail(c, RT_EINVAL, "groups must be in [0, %d]", kSlots);
    c->groups_req = groups;
    return RT_OK;
}

int rt_set_block_threads(rt_ctx* c, int threads)
{
    int rc = enter(c);
    if (rc) return rc;
    if (threads != 0 && threads != 64 && threads != 128 && threads != 256)
        return fail(c, RT_EINVAL, "threads per block must be 0 (default), 64, 128 or 256");
    c->threads32 = threads;
    return RT_OK;
}

int rt_set_block_order(rt_ctx* c, int order)
{
    int rc = enter(c);
    if (rc) return rc;
    if (order < 0 || order > 2)
        return fail(c, RT_EINVAL, "block order must be 0 (automatic), 1 (tile-major) or 2 (plane-major)");
    c->order32 = order;
    return RT_OK;
}

int rt_set_cutoff(rt_ctx* c, double cut)
{
    if (!c) return RT_EINVAL;
    if (!(cut >= 0) || !(cut < 1)) return fail(c, RT_EINVAL, "cutoff must lie in [0, 1)");
    c->cut = cut;
    c->rec_valid = false;
    return RT_OK;
}

int rt_set_fs_record(rt_ctx* c, long long max_bytes)
{
    int rc = enter(c);
    if (rc) return rc;
    if (max_bytes < -1) return fail(c, RT_EINVAL, "max_bytes must be -1 (automatic), 0 (off) or a byte limit");
    CK(cudaStreamSynchronize(c->stream));
    c->rec_mode = max_bytes;
    if (max_bytes >= 0 && c->rec_cap > max_bytes) free_rec(c);
    c->rec_valid = false;
    return RT_OK;
}

int rt_fs_record_info(rt_ctx* c, long long* bytes, int* valid)
{
    if (!c || !bytes || !valid) return RT_EINVAL;
    *bytes = c->rec_cap;
    *valid = c->rec_valid ? 1 : 0;
    return RT_OK;
}

int rt_segment_weights(int precision, long long n, const double* x, double* w_cur, double* w_up,
                       double* e, void* stream)
{
    if (n < 0 || (n > 0 && (!x || !w_cur || !w_up || !e))) return RT_EINVAL;
    if (precision != RT_FP64 && precision != RT_FP32_SWEEP) return RT_EINVAL;
    if (n == 0) return RT_OK;
    if (launch_seg_eval(n, precision == RT_FP32_SWEEP, x, w_cur, w_up, e, (cudaStream_t)stream) !=
        cudaSuccess)
        return RT_ECUDA;
    return RT_OK;
}

int rt_set_ng(rt_ctx* c, int period, double min_delta)
{
    if (!c) return RT_EINVAL;
    if (period != 0 && period < 4) return fail(c, RT_EINVAL, "Ng period must be 0 (off) or >= 4");
    if (!(min_delta >= 0)) return fail(c, RT_EINVAL, "Ng min_delta must be >= 0");
    c->ng_period = period;
    c->ng_min_delta = min_delta;
    c->ng_count = 1;
    return RT_OK;
}

int rt_set_fs_method(rt_ctx* c, int method)
{
    if (!c) return RT_EINVAL;
    if (method != RT_FS_LONG && method != RT_FS_SHORT)
        return fail(c, RT_EINVAL, "unknown formal-solution method");
    if (method == RT_FS_SHORT && c->precision != RT_FP64 && c->precision != RT_DF64)
        return fail(c, RT_EINVAL, "short characteristics need precision RT_FP64 or RT_DF64");
    if (method == RT_FS_SHORT && c->src_order != RT_SRC_LINEAR)
        return fail(c, RT_EINVAL, "short characteristics take the linear source only");
    if (method != c->fs_method) {
        c->fs_method = method;
        c->lstar_valid = c->coef_valid = c->rec_valid = false;   // Lambda* differs between methods
    }
    return RT_OK;
}

int rt_set_precision(rt_ctx* c, int precision)
{
    int rc = enter(c);
    if (rc) return rc;
    return switch_precision(c, precision);
}


int rt_set_graphs(rt_ctx* c, int on)
{
    if (!c) return RT_EINVAL;
    c->use_graphs = on != 0;
    return RT_OK;
}

int rt_set_df_finish(rt_ctx* c, double delta_switch)
{
    if (!c) return RT_EINVAL;
    if (!(delta_switch >= 0)) return fail(c, RT_EINVAL, "delta_switch must be >= 0");
    c->df_switch = delta_switch;
    return RT_OK;
}

int rt_batch_set_df_finish(rt_batch* b, double delta_switch)
{
    if (!b) return RT_EINVAL;
    if (!(delta_switch >= 0)) return bfail(b, RT_EINVAL, "delta_switch must be >= 0");
    for (rt_ctx* c : b->ctx) c->df_switch = delta_switch;
    return RT_OK;
}

int rt_set_source_order(rt_ctx* c, int order)
{
    if (!c) return RT_EINVAL;
    if (order != RT_SRC_LINEAR && order != RT_SRC_PARABOLIC)
        return fail(c, RT_EINVAL, "unknown source order");
    if (order == RT_SRC_PARABOLIC && (c->precision != RT_FP64 || c->fs_method != RT_FS_LONG))
        return fail(c, RT_EINVAL, "the parabolic source needs RT_FP64 and long characteristics");
    if (order != c->src_order) {
        c->src_order = order;
        c->lstar_valid = c->coef_valid = c->rec_valid = false;
    }
    return RT_OK;
}

int rt_set_os_method(rt_ctx* c, int method)
{
    if (!c) return RT_EINVAL;
    if (method != RT_OS_JACOBI && method != RT_OS_GAUSS_SEIDEL)
        return fail(c, RT_EINVAL, "unknown operator-splitting method");
    if (method != c->os_method) {
        c->os_method = method;
        c->coef_valid = false;   // the storage of c, 1/diag, r differs
    }
    return RT_OK;
}

int rt_batch_set_os_method(rt_batch* b, int method)
{
    if (!b) return RT_EINVAL;
    if (method != RT_OS_JACOBI && method != RT_OS_GAUSS_SEIDEL)
        return bfail(b, RT_EINVAL, "unknown operator-splitting method");
    for (rt_ctx* c : b->ctx) rt_set_os_method(c, method);
    return RT_OK;
}

int rt_batch_set_ng(rt_batch* b, int period, double min_delta)
{
    if (!b) return RT_EINVAL;
    if (period != 0 && period < 4) return bfail(b, RT_EINVAL, "Ng period must be 0 (off) or >= 4");
    if (!(min_delta >= 0)) return bfail(b, RT_EINVAL, "Ng min_delta must be >= 0");
    for (rt_ctx* c : b->ctx) rt_set_ng(c, period, min_delta);
    return RT_OK;
}

int rt_set_profiling(rt_ctx* c, int on)
{
    if (!c) return RT_EINVAL;
    c->profiling = on != 0;
    return RT_OK;
}

int rt_get_stats(rt_ctx* c, rt_stats* out)
{
    if (!c || !out) return RT_EINVAL;
    *out = c->stats;
    return RT_OK;
}

int rt_reset_stats(rt_ctx* c)
{
    if (!c) return RT_EINVAL;
    c->stats = rt_stats{};
    return RT_OK;
}

// ---- batched wavelengths (C ABI) --------------------------------------------

int rt_batch_create(rt_batch** out, int device, int precision, int nprob, const rt_problem* probs,
                    int top_mode, int bottom_mode, int ndir, const double* mu, const double* phi,
                    const double* w)
{
    if (!out) return RT_EINVAL;
    *out = nullptr;
    if (nprob < 1 || !probs ||
        (precision != RT_FP64 && precision != RT_FP32_SWEEP && precision != RT_DF64))
        return RT_EINVAL;
    rt_batch* b = new rt_batch();
    b->device = device;
    b->precision = precision;
    *out = b;  // also on failure, for rt_batch_last_error; the caller destroys it
    int rc = RT_OK;
    auto bail = [&](int code) { return code; };
    if (cudaSetDevice(device) != cudaSuccess ||
        cudaStreamCreateWithFlags(&b->own_stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaDeviceGetAttribute(&b->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
        return bail(bfail(b, RT_ECUDA, "device %d unavailable", device));
    b->stream = b->own_stream;
    for (int e = 0; e < 4; ++e) BCK(cudaEventCreate(&b->ev[e]));
    b->ctx.assign(nprob, nullptr);
    for (int p = 0; p < nprob; ++p) {
        const rt_problem& q = probs[p];
        rt_ctx* c = nullptr;
        if ((rc = rt_create(&c, device, precision))) return bail(bfail(b, rc, "problem %d: context", p));
        b->ctx[p] = c;
        if ((rc = rt_set_stream(c, b->stream)) || (rc = rt_set_grid(c, q.nx, q.ny, q.nz, q.dx, q.dy, q.dz)) ||
            (rc = rt_set_boundary(c, top_mode, bottom_mode)) ||
            (rc = rt_set_quadrature(c, ndir, mu, phi, w)) || (rc = rt_set_opacity(c, q.chi)) ||
            (rc = rt_set_epsilon(c, q.eps)) || (rc = rt_set_planck(c, q.B)) ||
            (rc = ensure_partial(c)))
            return bail(bpass(b, p, rc));
    }
    b->order.resize(nprob);
    for (int p = 0; p < nprob; ++p) b->order[p] = p;
    std::stable_sort(b->order.begin(), b->order.end(),
                     [&](int x, int y) { return b->ctx[x]->g.N > b->ctx[y]->g.N; });
    b->iters.assign(nprob, 0);
    b->delta.assign(nprob, 0.0);
    b->converged.assign(nprob, 0);
    b->admitted.assign(nprob, 0);
    BCK(cudaMallocHost((void**)&b->h_views, sizeof(View32) * nprob));
    for (int p = 0; p < nprob; ++p) b->h_views[p] = view32(b->ctx[p]);
    b->view_fin.assign(nprob, 0);
    BCK(cudaMalloc((void**)&b->d_views, sizeof(View32) * nprob));
    BCK(cudaMemcpy(b->d_views, b->h_views, sizeof(View32) * nprob, cudaMemcpyHostToDevice));
    BCK(cudaMalloc((void**)&b->d_ids, sizeof(int) * nprob));
    BCK(cudaMalloc((void**)&b->d_prefix, sizeof(long long) * (nprob + 1)));
    BCK(cudaMalloc((void**)&b->d_delta, sizeof(double) * nprob));
    BCK(cudaMalloc((void**)&b->d_steps, sizeof(unsigned long long)));
    BCK(cudaMallocHost((void**)&b->h_ids, sizeof(int) * nprob));
    BCK(cudaMalloc((void**)&b->d_rviews, sizeof(Rep32) * nprob));
    BCK(cudaMallocHost((void**)&b->h_rviews, sizeof(Rep32) * nprob));
    memset(b->h_rviews, 0, sizeof(Rep32) * nprob);
    BCK(cudaMalloc((void**)&b->d_rids, sizeof(int) * nprob));
    BCK(cudaMalloc((void**)&b->d_rprefix, sizeof(long long) * (nprob + 1)));
    BCK(cudaMallocHost((void**)&b->h_rids, sizeof(int) * nprob));
    BCK(cudaMallocHost((void**)&b->h_rprefix, sizeof(long long) * (nprob + 1)));
    BCK(cudaMallocHost((void**)&b->h_prefix, sizeof(long long) * (nprob + 1)));
    BCK(cudaMallocHost((void**)&b->h_delta, sizeof(double) * nprob));
    BCK(cudaMallocHost((void**)&b->h_steps, sizeof(unsigned long long)));
    BCK(cudaMalloc((void**)&b->d_sweeps, sizeof(int) * nprob));
    BCK(cudaMemset(b->d_sweeps, 0, sizeof(int) * nprob));
    BCK(cudaMallocHost((void**)&b->h_sweeps, sizeof(int) * nprob));
    *out = b;
    return RT_OK;
}

int rt_batch_destroy(rt_batch* b)
{
    if (!b) return RT_OK;
    cudaSetDevice(b->device);
    if (b->stream) cudaStreamSynchronize(b->stream);
    free_batch_graphs(b);
    batch_free_pool(b);
    for (rt_ctx* c : b->ctx) rt_destroy(c);
    if (b->d_tasks) cudaFree(b->d_tasks);
    if (b->d_first) cudaFree(b->d_first);
    if (b->h_tasks) cudaFreeHost(b->h_tasks);
    if (b->h_first) cudaFreeHost(b->h_first);
    if (b->d_bdlt) cudaFree(b->d_bdlt);
    if (b->d_sweeps) cudaFree(b->d_sweeps);
    if (b->h_sweeps) cudaFreeHost(b->h_sweeps);
    if (b->d_views) cudaFree(b->d_views);
    if (b->h_views) cudaFreeHost(b->h_views);
    if (b->d_rviews) cudaFree(b->d_rviews);
    if (b->h_rviews) cudaFreeHost(b->h_rviews);
    if (b->d_rids) cudaFree(b->d_rids);
    if (b->d_rprefix) cudaFree(b->d_rprefix);
    if (b->h_rids) cudaFreeHost(b->h_rids);
    if (b->h_rprefix) cudaFreeHost(b->h_rprefix);
    if (b->d_ids) cudaFree(b->d_ids);
    if (b->d_prefix) cudaFree(b->d_prefix);
    if (b->d_delta) cudaFree(b->d_delta);
    if (b->d_steps) cudaFree(b->d_steps);
    if (b->h_ids) cudaFreeHost(b->h_ids);
    if (b->h_prefix) cudaFreeHost(b->h_prefix);
    if (b->h_delta) cudaFreeHost(b->h_delta);
    if (b->h_steps) cudaFreeHost(b->h_steps);
    for (auto& e : b->ev)
        if (e) cudaEventDestroy(e);
    if (b->own_stream) cudaStreamDestroy(b->own_stream);
    delete b;
    return RT_OK;
}

const char* rt_batch_last_error(const rt_batch* b) { return b ? b->err.c_str() : "null batch"; }

int rt_batch_set_stream(rt_batch* b, void* stream)
{
    if (!b) return RT_EINVAL;
    b->err.clear();
    BCK(cudaSetDevice(b->device));
    BCK(cudaStreamSynchronize(b->stream));
    b->stream = stream ? (cudaStream_t)stream : b->own_stream;
    free_batch_graphs(b);
    for (size_t p = 0; p < b->ctx.size(); ++p) {
        int rc = rt_set_stream(b->ctx[p], b->stream);
        if (rc) return bpass(b, (int)p, rc);
    }
    return RT_OK;
}

int rt_batch_reset(rt_batch* b, int rebuild_lstar)
{
    if (!b) return RT_EINVAL;
    b->err.clear();
    BCK(cudaSetDevice(b->device));
    for (size_t p = 0; p < b->ctx.size(); ++p) {
        rt_ctx* c = b->ctx[p];
        BCK(cudaMemcpyAsync(c->J, c->B, sizeof(double) * c->g.N, cudaMemcpyDeviceToDevice,
                            b->stream));
        c->ng_count = 1;
        c->ng_last_delta = 0.0;
        if (rebuild_lstar) c->lstar_valid = c->coef_valid = false;
        b->iters[p] = 0;
        b->delta[p] = 0.0;
        b->converged[p] = 0;
        b->admitted[p] = c->rec_cap > 0;   // a held recording keeps its place
    }
    return RT_OK;
}

int rt_batch_set_fs_record(rt_batch* b, long long max_bytes)
{
    if (!b) return RT_EINVAL;
    b->err.clear();
    if (max_bytes < -1) return bfail(b, RT_EINVAL, "max_bytes must be -1 (automatic), 0 (off) or a byte limit");
    BCK(cudaSetDevice(b->device));
    for (size_t p = 0; p < b->ctx.size(); ++p) batch_release(b, (int)p);
    batch_free_pool(b);
    std::fill(b->admitted.begin(), b->admitted.end(), 0);
    b->rec_mode = max_bytes;
    return RT_OK;
}

int rt_batch_set_precision(rt_batch* b, int precision)
{
    if (!b) return RT_EINVAL;
    b->err.clear();
    BCK(cudaSetDevice(b->device));
    if (precision == b->precision) return RT_OK;
    if (!((precision == RT_FP32_SWEEP || precision == RT_DF64) &&
          (b->precision == RT_FP32_SWEEP || b->precision == RT_DF64)))
        return bfail(b, RT_EINVAL, "precision switches only between RT_FP32_SWEEP and RT_DF64");
    for (size_t p = 0; p < b->ctx.size(); ++p) {
        const int rc = rt_set_precision(b->ctx[p], precision);
        if (rc) return bfail(b, rc, "problem %zu: %s", p, rt_last_error(b->ctx[p]));
        b->iters[p] = 0;        // a new stage: counts, deltas and convergence restart
        b->delta[p] = 0.0;
        b->converged[p] = 0;
        batch_release(b, (int)p);
        b->admitted[p] = 0;
    }
    batch_free_pool(b);
    b->precision = precision;
    return RT_OK;
}

static int batch_solve(rt_batch* b, double tol, int max_iter, double tol_inner, int max_sweeps,
                       int* iters, double* deltas, int* n_converged);

int rt_batch_solve(rt_batch* b, double tol, int max_iter, double tol_inner, int max_sweeps,
                   int* iters, double* deltas, int* n_converged)
{
    int rc = batch_solve(b, tol, max_iter, tol_inner, max_sweeps, iters, deltas, n_converged);
    if (!b) return rc;
    for (size_t p = 0; p < b->ctx.size(); ++p) {
        const int r2 = check_bounds(b->ctx[p], RT_OK);
        if (r2) return bfail(b, r2, "problem %zu: %s", p, rt_last_error(b->ctx[p]));
    }
    return rc;
}

int rt_checked_build(void)
{
#ifdef RT_CHECKED
    return 1;
#else
    return 0;
#endif
}

int rt_bounds_selftest(rt_ctx* c)
{
    int rc = enter(c);
    if (rc) return rc;
    CK(launch_bounds_selftest(c->g, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    return check_bounds(c, RT_OK);
}

int rt_get_plane_order(rt_ctx* c, int* order)
{
    int rc = enter(c);
    if (rc) return rc;
    if ((rc = need(c, c->have_chi, "the opacity"))) return rc;
    if (!order) return fail(c, RT_EINVAL, "order is NULL");
    CK(cudaMemcpyAsync(order, c->zorder, sizeof(int) * c->g.nz, cudaMemcpyDeviceToHost,
                       c->stream));
    CK(cudaStreamSynchronize(c->stream));
    return RT_OK;
}

static int batch_solve(rt_batch* b, double tol, int max_iter, double tol_inner, int max_sweeps,
                       int* iters, double* deltas, int* n_converged)
{
    if (!b) return RT_EINVAL;
    b->err.clear();
    BCK(cudaSetDevice(b->device));
    if (max_iter < 1 || max_sweeps < 1 || !(tol >= 0) || !(tol_inner >= 0))
        return bfail(b, RT_EINVAL, "bad iteration controls");
    const int P = (int)b->ctx.size();
    int rc;
    // problems in their finishing stage leave it (and get their Ng threshold
    // back) when the solve ends, whichever way it ends
    struct FinishGuard {
        rt_batch* b;
        std::vector<char> switched;
        std::vector<double> ng_min0;
        ~FinishGuard()
        {
            for (size_t p = 0; p < switched.size(); ++p)
                if (switched[p]) {
                    b->ctx[p]->fin = 0;
                    b->ctx[p]->ng_min_delta = ng_min0[p];
                }
        }
    } guard{b, std::vector<char>(P, 0), std::vector<double>(P, 0.0)};
    std::vector<char>& switched = guard.switched;
    std::vector<double>& ng_min0 = guard.ng_min0;
    // (problems admitted in waves: the loop runs until none is left)
    for (long long it = 0; it < (long long)max_iter * P + 1; ++it) {
        if ((rc = batch_admit(b, max_iter))) return rc;
        std::vector<int> act;
        for (int p : b->order)
            if (b->admitted[p] && !b->converged[p] && b->iters[p] < max_iter) act.push_back(p);
        if (act.empty()) break;
        if ((rc = batch_fs(b, act))) return rc;
        BCK(cudaMemsetAsync(b->d_delta, 0, sizeof(double) * P, b->stream));
        std::vector<double*> hist(P, nullptr);
        std::vector<char> due(P, 0);
        rc = RT_OK;
        for (int p : act) {
            bool d = false;
            if ((rc = bpass(b, p, ng_begin(b->ctx[p], b->iters[p] + 1, b->d_delta + p, hist[p], d)))) break;
            due[p] = d;
        }
        b->os_one = false;
        if (rc == RT_OK)
            rc = b->use_graphs ? batch_os_graph(b, act, tol_inner, max_sweeps)
                               : batch_os(b, act, tol_inner, max_sweeps);
        if (rc) {
            for (int p : act) ng_forget(b->ctx[p]);
            return rc;
        }
        for (int p : act) {
            if ((rc = bpass(b, p, ng_end(b->ctx[p], b->os_one, due[p], b->d_delta + p, hist[p])))) return rc;
            b->stats.launches += b->os_one && !due[p] ? 0 : 1;
        }
        BCK(cudaMemcpyAsync(b->h_delta, b->d_delta, sizeof(double) * P, cudaMemcpyDeviceToHost,
                            b->stream));
        if (b->use_graphs)
            BCK(cudaMemcpyAsync(b->h_sweeps, b->d_sweeps, sizeof(int) * P, cudaMemcpyDeviceToHost,
                                b->stream));
        BCK(cudaStreamSynchronize(b->stream));
        b->stats.host_syncs += 1;
        b->stats.iterations += 1;
        if (b->use_graphs && (rc = batch_os_graph_counts(b, act))) {
            for (int p : act) ng_forget(b->ctx[p]);     // histories may not have been written
            return rc;
        }
        bharvest(b);
        b->stats.steps += *b->h_steps;
        for (int p : act) {
            rt_ctx* c = b->ctx[p];
            std::swap(c->J, c->Jn);
            b->iters[p] += 1;
            b->delta[p] = b->h_delta[p];
            c->ng_last_delta = b->h_delta[p];
            if (tol > 0 && b->h_delta[p] < tol) {
                b->converged[p] = 1;
            } else if (c->df_switch > 0 && c->precision == RT_FP32_SWEEP &&
                       b->precision == RT_FP32_SWEEP && c->fin == 0 &&
                       b->h_delta[p] < c->df_switch) {
                // finishing stage for this problem (see solve())
                c->fin = 1;
                switched[p] = 1;
                ng_min0[p] = c->ng_min_delta;
                c->ng_min_delta = 0.0;
                c->ng_count = 1;
            }
            if (b->converged[p] || b->iters[p] >= max_iter) {
                batch_release(b, p);
                b->admitted[p] = 0;             // a later solve admits it again
            }
        }
    }
    batch_free_pool(b, kPoolKeep);
    int nconv = 0;
    for (int p = 0; p < P; ++p) {
        if (iters) iters[p] = b->iters[p];
        if (deltas) deltas[p] = b->delta[p];
        nconv += b->converged[p];
    }
    if (n_converged) *n_converged = nconv;
    if (tol > 0 && nconv < P)
        return bfail(b, RT_ENOTCONV, "%d of %d problems not converged", P - nconv, P);
    return RT_OK;
}

int rt_batch_get_J(rt_batch* b, int p, double* J)
{
    if (!b || !J || p < 0 || p >= (int)b->ctx.size()) return RT_EINVAL;
    b->err.clear();
    BCK(cudaSetDevice(b->device));
    BCK(cudaStreamSynchronize(b->stream));
    int rc = rt_get_J(b->ctx[p], J);
    return bpass(b, p, rc);
}

int rt_batch_get_J_dev(rt_batch* b, int p, double* J)
{
    if (!b || !J || p < 0 || p >= (int)b->ctx.size()) return RT_EINVAL;
    b->err.clear();
    BCK(cudaSetDevice(b->device));
    rt_ctx* c = b->ctx[p];
    BCK(cudaMemcpyAsync(J, c->J, sizeof(double) * c->g.N, cudaMemcpyDeviceToDevice, b->stream));
    return RT_OK;
}

int rt_batch_set_block_threads(rt_batch* b, int threads)
{
    if (!b) return RT_EINVAL;
    if (threads != 0 && threads != 64 && threads != 128 && threads != 256)
        return bfail(b, RT_EINVAL, "threads per block must be 0 (default), 64, 128 or 256");
    b->threads32 = threads;
    return RT_OK;
}

int rt_batch_set_block_order(rt_batch* b, int order)
{
    if (!b) return RT_EINVAL;
    b->err.clear();
    if (order < 0 || order > 2)
        return bfail(b, RT_EINVAL, "block order must be 0 (automatic), 1 (tile-major) or 2 (plane-major)");
    for (rt_ctx* c : b->ctx) c->order32 = order;
    const int n = (int)b->ctx.size();
    for (int p = 0; p < n; ++p)
        b->h_views[p] = b->view_fin[p] ? view32_fin(b->ctx[p]) : view32(b->ctx[p]);
    BCK(cudaMemcpyAsync(b->d_views, b->h_views, sizeof(View32) * n, cudaMemcpyHostToDevice,
                        b->stream));
    BCK(cudaStreamSynchronize(b->stream));
    return RT_OK;
}

int rt_batch_set_graphs(rt_batch* b, int on)
{
    if (!b) return RT_EINVAL;
    b->err.clear();
    BCK(cudaSetDevice(b->device));
    BCK(cudaStreamSynchronize(b->stream));
    free_batch_graphs(b);
    b->use_graphs = on != 0;
    return RT_OK;
}

int rt_batch_set_direction_groups(rt_batch* b, int groups)
{
    if (!b) return RT_EINVAL;
    if (groups < 0 || groups > kSlots) return bfail(b, RT_EINVAL, "groups must be in [0, %d]", kSlots);
    b->groups_req = groups;
    return RT_OK;
}

int rt_batch_set_profiling(rt_batch* b, int on)
{
    if (!b) return RT_EINVAL;
    b->profiling = on != 0;
    return RT_OK;
}

int rt_batch_get_stats(rt_batch* b, rt_stats* out)
{
    if (!b || !out) return RT_EINVAL;
    rt_stats s = b->stats;
    for (rt_ctx* c : b->ctx) {   // per-problem kernels (source, sums, Lambda*, OS set-up)
        s.launches += c->stats.launches;
        s.lstar_launches += c->stats.lstar_launches;
    }
    *out = s;
    return RT_OK;
}

int rt_batch_reset_stats(rt_batch* b)
{
    if (!b) return RT_EINVAL;
    b->stats = rt_stats{};
    for (rt_ctx* c : b->ctx) c->stats = rt_stats{};
    return RT_OK;
}

}  // extern "C"
