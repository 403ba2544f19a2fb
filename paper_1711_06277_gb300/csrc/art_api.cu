// art_api.cu -- C ABI of the GB300 adaptive ray trace: grid object, argument checks,
// buffer management and the launch sequences of the forward trace.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "art.h"
#include "art_kernels.cuh"
#include "art_internal.h"

using namespace art;

namespace {

constexpr double kDefaultWaitS = 60.0;

int cuda_status(cudaError_t e)
{
    if (e == cudaSuccess) return ART_OK;
    if (e == cudaErrorMemoryAllocation) return ART_ENOMEM;
    return ART_ECUDA;
}

#define ART_TRY(expr)                     \
    do {                                  \
        int _rc = cuda_status(expr);      \
        if (_rc != ART_OK) return _rc;    \
    } while (0)

double rmax_unit(double m_ray) { return std::sqrt(3.0 / (M_PI * m_ray)); }

// l_max of a source at u (cell units): smallest l >= l0 whose split radius reaches the
// farthest corner of the box, capped at ART_MAX_LEVEL; or the fixed cap.
int source_level_max(const art_grid* g, const double u[3], int level0, int cap, double m_ray)
{
    if (cap >= 0) return cap;
    double far2 = 0.0;
    for (int a = 0; a < 3; ++a) {
        double e = std::fmax(u[a], (double)g->n[a] - u[a]);
        far2 += e * e;
    }
    const double far = std::sqrt(far2);
    const double unit = rmax_unit(m_ray);
    int l = level0;
    while (l < ART_MAX_LEVEL && unit * std::ldexp(1.0, l) < far) ++l;
    return l;
}

void split_df(double v, float& hi, float& lo)
{
    hi = (float)v;
    lo = (float)(v - (double)hi);
}

using LevelKernel = void (*)(TraceArgs, int, unsigned);
using PersistentKernel = void (*)(TraceArgs);

// The kernels for one or two bins, with or without a cutoff and a force.
template <class Cell>
LevelKernel level_kernel_of(bool cut, bool force)
{
    return cut ? (force ? k_trace_level<Cell, true, true> : k_trace_level<Cell, true, false>)
               : (force ? k_trace_level<Cell, false, true> : k_trace_level<Cell, false, false>);
}
LevelKernel level_kernel(bool two_bin, bool cut, bool force)
{
    return two_bin ? level_kernel_of<float2>(cut, force) : level_kernel_of<float>(cut, force);
}
template <class Cell>
PersistentKernel persistent_kernel_of(bool cut, bool force)
{
    return cut ? (force ? k_trace_persistent<Cell, true, true> : k_trace_persistent<Cell, true, false>)
               : (force ? k_trace_persistent<Cell, false, true> : k_trace_persistent<Cell, false, false>);
}
PersistentKernel persistent_kernel(bool two_bin, bool cut, bool force)
{
    return two_bin ? persistent_kernel_of<float2>(cut, force) : persistent_kernel_of<float>(cut, force);
}

template <class T>
int dev_alloc(T** p, size_t count)
{
    *p = nullptr;
    if (count == 0) count = 1;
    return cuda_status(cudaMalloc((void**)p, count * sizeof(T)));
}

void dev_free(void* p)
{
    if (p) cudaFree(p);
}

void free_retired(art_grid* g)
{
    for (void* p : g->retired) dev_free(p);
    g->retired.clear();
}

}  // namespace

// ---------------------------------------------------------------------------------------
// shared helpers (declared in art_internal.h)
// ---------------------------------------------------------------------------------------
namespace art {

int check_params(const art_params* p)
{
    if (!p) return ART_EINVAL;
    if (p->level0 < 0 || p->level0 > 12) return ART_EINVAL;
    if (p->level_max >= 0 && (p->level_max < p->level0 || p->level_max > ART_MAX_LEVEL))
        return ART_EINVAL;
    if (!(p->m_ray > 0.0) || !std::isfinite(p->m_ray)) return ART_EINVAL;
    if (!(p->tau_max > 0.0) || !(p->tau_max < 3.0e38)) return ART_EINVAL;
    if (!(p->sigma_H >= 0.0) || !(p->sigma_d >= 0.0) || !std::isfinite(p->sigma_H) ||
        !std::isfinite(p->sigma_d))
        return ART_EINVAL;
    if (p->schedule != ART_SCHED_PERSISTENT && p->schedule != ART_SCHED_PLAIN) return ART_EINVAL;
    if (p->block_threads != 0 &&
        (p->block_threads % 32 != 0 || p->block_threads < 64 || p->block_threads > 1024))
        return ART_EINVAL;
    if (p->chunk != 0 && (p->chunk < 32 || p->chunk % 32 != 0)) return ART_EINVAL;
    if (p->queue_capacity != 0 && (p->queue_capacity < 4 || p->queue_capacity > (1ll << 30)))
        return ART_EINVAL;
    if (p->blocks_per_sm < 0) return ART_EINVAL;
    if (p->d_max != p->d_max || (p->d_max > 0.0 && !std::isfinite(p->d_max))) return ART_EINVAL;
    if (p->flags & ART_F_ROTATE)
        for (int i = 0; i < 9; ++i)
            if (!std::isfinite(p->rot[i])) return ART_EINVAL;
    return ART_OK;
}

// Split radius r_max(l) = [3/(pi m_ray)]^(1/2) 2^l in cells (Sec. 2.1).
double rmax_cells(double m_ray, int level) { return rmax_unit(m_ray) * std::ldexp(1.0, level); }

// A distance in cells as a fixed-point number; distances beyond every box (radii of levels
// that no ray reaches) end up just below kFar.
fix to_fix(double cells, int fbits)
{
    const double v = std::ldexp(cells, fbits);
    return v < (double)kFar ? (fix)std::llrint(v) : kFar - 1;
}

// An opacity coefficient for the device: two floats where products with densities below 1e18
// stay in their range, parts included.
Coef coef_of(double v)
{
    Coef c;
    split_df(v, c.hi, c.lo);
    c.full = v;
    c.wide = v != 0.0 && !(v > 1e-18 && v < 1e18);
    return c;
}

// Device record of a source at u (cell units).
SrcDev source_record(const art_grid* g, const double u[3], double base_L, int lmax)
{
    SrcDev d;
    float h[3], lo[3], lmf;
    for (int a = 0; a < 3; ++a) split_df(u[a], h[a], lo[a]);
    std::memcpy(&lmf, &lmax, sizeof(float));
    d.hi = make_float4(h[0], h[1], h[2], (float)base_L);
    d.lo = make_float4(lo[0], lo[1], lo[2], lmf);
    d.xy = make_longlong2(to_fix(u[0], g->fbits), to_fix(u[1], g->fbits));
    d.z_ = make_longlong2(to_fix(u[2], g->fbits),
                          pad_index((long long)u[0], (long long)u[1], (long long)u[2], g->n[0], g->n[1]));
    return d;
}

// Direction tables of levels lfrom..lto (FP64 HEALPix, rotated by p's rotation, split
// into hi + lo), rebuilt when the rotation changes.
int ensure_directions(art_grid* g, const art_params* p, int lfrom, int lto)
{
    const bool rotate = (p->flags & ART_F_ROTATE) != 0;
    bool same_rot = g->dir_rotate == rotate;
    if (rotate && same_rot)
        for (int i = 0; i < 9; ++i) same_rot = same_rot && g->dir_rot[i] == p->rot[i];
    if (!same_rot) {
        for (int l = 0; l < kNL; ++l) g->dir_built[l] = false;
        g->dir_rotate = rotate;
        for (int i = 0; i < 9; ++i) g->dir_rot[i] = rotate ? p->rot[i] : (i % 4 == 0 ? 1.0 : 0.0);
    }
    for (int l = lfrom; l <= lto; ++l) {
        const unsigned long long npix = 12ull << (2 * l);
        if (!g->dir[l]) {
            int rc = dev_alloc(&g->dir[l], 3 * npix);
            if (rc) return rc;
            g->dir_built[l] = false;
        }
        if (!g->dir_built[l]) {
            const double* r = g->dir_rot;
            unsigned blocks = (unsigned)((npix + 255) / 256);
            k_directions<<<blocks, 256, 0, g->stream>>>(l, npix, r[0], r[1], r[2], r[3], r[4],
                                                        r[5], r[6], r[7], r[8], rotate ? 1 : 0,
                                                        std::ldexp(1.0, g->fbits), g->dir[l]);
            ART_TRY(cudaGetLastError());
            g->dir_built[l] = true;
        }
    }
    return ART_OK;
}

// Front of level l with room for `need` quads of a reverse sweep.
static int ensure_adjoint_front(art_grid* g, int l, unsigned long long need)
{
    AdjBuf& b = g->adj[l];
    if (need > g->adj_cap[l]) {
        dev_free(b.rec); dev_free(b.parent); dev_free(b.own); dev_free(b.sub);
        b = AdjBuf{};
        g->adj_cap[l] = 0;
        int rc = dev_alloc(&b.rec, need);
        if (!rc) rc = dev_alloc(&b.parent, need);
        if (!rc) rc = dev_alloc(&b.own, 4 * need);
        if (!rc) rc = dev_alloc(&b.sub, 4 * need);
        if (rc) return rc;
        g->adj_cap[l] = need;
    }
    b.cap = need;  // the capacity this sweep may use
    return ART_OK;
}

// Front of level l with room for `need` quads of a forward trace.
static int ensure_quads(art_grid* g, int l, unsigned long long need, bool two_bin)
{
    QuadBuf& q = g->quad[l];
    if (need > g->quad_cap[l]) {
        dev_free(q.rec);
        dev_free(q.recn);
        q = QuadBuf{};
        g->quad_cap[l] = 0;
        const int rc = dev_alloc(&q.rec, need);
        if (rc) return rc;
        g->quad_cap[l] = need;
    }
    if (two_bin && !q.recn) {
        const int rc = dev_alloc(&q.recn, g->quad_cap[l]);
        if (rc) return rc;
    }
    q.cap = need;  // the capacity this trace may use
    return ART_OK;
}

// Words of a table that travel as a kernel's parameter.
template <int kWords>
struct Words {
    uint4 w[kWords];
};
template <int kWords>
__global__ void k_store(const __grid_constant__ Words<kWords> from, uint4* __restrict__ to, unsigned n)
{
    for (unsigned i = threadIdx.x; i < n; i += blockDim.x) to[i] = from.w[i];
}
template <int kWords>
static cudaError_t store_words(const unsigned char* from, size_t bytes, uint4* to, cudaStream_t st)
{
    Words<kWords> w;
    std::memcpy(w.w, from, bytes);
    k_store<kWords><<<1, 64, 0, st>>>(w, to, (unsigned)(bytes / sizeof(uint4)));
    return cudaGetLastError();
}

// Brings a table of the device up to date. An unchanged one enqueues nothing (such a trace can be
// captured in a graph without it). The bytes travel as kernel parameters, which the launch
// takes over: a staging buffer may be written again while an earlier copy from it still waits in
// the stream, and a graph would read it at every replay.
static int send_table(art_grid* g, HostTable& t, const void* data, size_t bytes, void* to)
{
    const unsigned char* from = static_cast<const unsigned char*>(data);
    if (t.known && t.sent.size() == bytes && std::memcmp(t.sent.data(), from, bytes) == 0) return ART_OK;
    t.known = false;
    constexpr int kSmall = 64, kLarge = 1024;  // words of 16 bytes
    for (size_t at = 0; at < bytes;) {
        uint4* const dst = reinterpret_cast<uint4*>(static_cast<unsigned char*>(to) + at);
        const bool small = bytes - at <= kSmall * sizeof(uint4);
        const size_t n = std::min(bytes - at, kLarge * sizeof(uint4));
        ART_TRY(small ? store_words<kSmall>(from + at, n, dst, g->stream)
                      : store_words<kLarge>(from + at, n, dst, g->stream));
        at += n;
    }
    // captured into a graph, the table changes whenever the graph runs: no call can tell any more
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    ART_TRY(cudaStreamIsCapturing(g->stream, &cs));
    t.in_graph = t.in_graph || cs != cudaStreamCaptureStatusNone;
    if (!t.in_graph) {
        t.sent.assign(from, from + bytes);
        t.known = true;
    }
    return ART_OK;
}

// Source table, per-source l_max, direction tables, level constants and ray buffers for a
// trace with parameters p. Allocates only when something grew or changed.
int prepare_trace(art_grid* g, const art_params* p, bool adjoint)
{
    const int ns = (int)g->L.size();
    if (ns == 0) return ART_ESTATE;
    const int l0 = p->level0;
    const unsigned npix0 = 12u << (2 * l0);
    if ((unsigned long long)ns * npix0 >= (1ull << 31)) return ART_EINVAL;  // 32-bit ray slots
    // --- sources: cell-unit positions as df, base-ray luminosity, l_max
    std::vector<SrcDev> hs(ns);
    int lmax_glob = l0;
    g->src_lmax.resize(ns);
    for (int s = 0; s < ns; ++s) {
        double u[3];
        for (int a = 0; a < 3; ++a) u[a] = (g->pos[3 * s + a] - g->lo[a]) / g->dx;
        int lm = source_level_max(g, u, l0, p->level_max, p->m_ray);
        g->src_lmax[s] = lm;
        if (lm > lmax_glob) lmax_glob = lm;
        const double lb = adjoint ? 1.0 / (double)npix0 : g->L[s] / (double)npix0;
        hs[s] = source_record(g, u, lb, lm);
    }
    // The sums of first segments are kept for a fixed order of addition where base rays come in
    // whole groups of 64 of one source (from l0 = 2; every phase of the base front then ends on such
    // a group unless it is 16 quads or less, see below) and up to l0 = 6, 1536 sums per source: the
    // one warp that adds them takes longer beyond, and they are added as they come. They lie behind
    // the accumulator where they fit (creating and freeing a block of their own costs 0.3 ms from
    // 1 MB on), else in the allocation of the source table. A block of that which has become too
    // small for them alone may be in use by a captured trace and is kept.
    const size_t groups = !adjoint && l0 >= 2 && l0 <= 6 ? (size_t)ns * (npix0 / 32) : 0;
    const size_t own = groups * 8 <= g->first_room ? 0 : groups;
    SourceTables& T = g->tables[adjoint ? 1 : 0];
    if ((size_t)ns > T.cap || own > T.first_cap) {
        const size_t cap = (std::max((size_t)ns, T.cap) + 3) & ~(size_t)3;
        const size_t gcap = std::max(own, T.first_cap);
        if ((size_t)ns > T.cap) {
            dev_free(T.src);
            if (!adjoint) free_retired(g);
        } else {
            g->retired.push_back(T.src);
        }
        T = SourceTables{nullptr, nullptr, nullptr, nullptr, 0, 0, {}, {}, T.levels_sent};
        char* block = nullptr;
        const int rc = dev_alloc(&block, cap * (sizeof(SrcDev) + sizeof(double) + sizeof(float)) +
                                             gcap * 8 * sizeof(float4));
        if (rc) return rc;
        T.src = reinterpret_cast<SrcDev*>(block);
        T.first = reinterpret_cast<float*>(T.src + cap);
        T.dL = reinterpret_cast<double*>(T.first + gcap * 8 * 4);
        T.lum = reinterpret_cast<float*>(T.dL + cap);
        T.cap = cap;
        T.first_cap = gcap;
    }
    g->d_first = own ? T.first : reinterpret_cast<float*>(g->d_acc + g->npad);
    int rc = send_table(g, T.src_sent, hs.data(), ns * sizeof(SrcDev), T.src);
    if (rc) return rc;
    g->lmax_glob = lmax_glob;
    if (adjoint || g->two_bin) {
        std::vector<float> lum((ns + 3) & ~3, 0.f);  // whole words of 16 bytes
        for (int s = 0; s < ns; ++s) lum[s] = (float)(adjoint ? g->L[s] : g->Ln[s] / (double)npix0);
        if ((rc = send_table(g, T.lum_sent, lum.data(), lum.size() * sizeof(float), T.lum))) return rc;
    }
    if (g->two_bin && !adjoint && !g->d_chi2 && (rc = dev_alloc(&g->d_chi2, g->npad + 1))) return rc;
    // --- direction tables (FP64 HEALPix, rotated), rebuilt when the rotation changes
    if ((rc = ensure_directions(g, p, l0, lmax_glob))) return rc;
    // --- level constants
    static_assert(sizeof(SrcDev) % 16 == 0 && sizeof(LevelInfo) * kNL % 16 == 0, "stored in words");
    LevelInfo lv[kNL];
    std::memset(lv, 0, sizeof(lv));
    const double unit = rmax_unit(p->m_ray);
    for (int l = l0; l <= lmax_glob; ++l) {
        double r0 = l > l0 ? unit * std::ldexp(1.0, l - 1) : 0.0;
        double r1 = unit * std::ldexp(1.0, l);
        split_df(r0, lv[l].r0.hi, lv[l].r0.lo);
        lv[l].r0x = to_fix(r0, g->fbits);
        lv[l].rmaxx = to_fix(r1, g->fbits);
        lv[l].dir = g->dir[l];
        lv[l].destroy_w = 1ull << (2 * (lmax_glob - l));
    }
    if ((rc = send_table(g, T.levels_sent, lv, sizeof(lv), g->d_levels + (adjoint ? kNL : 0)))) return rc;
    // --- fronts: deeper levels hold at most the queue capacity (persistent) or one source's
    // whole front (plain); the base level of a forward trace needs no storage
    const bool plain = p->schedule == ART_SCHED_PLAIN;
    const long long qcap = p->queue_capacity > 0 ? p->queue_capacity : (64ll << 20);
    for (int l = l0; l <= lmax_glob; ++l) {
        unsigned long long need;
        const unsigned long long front = 12ull << (2 * l);  // rays of one source at level l
        if (l == l0) need = (unsigned long long)ns * npix0;
        else if (plain) need = p->queue_capacity > 0 ? (unsigned long long)qcap : front;
        else need = std::min<unsigned long long>((unsigned long long)qcap, (unsigned long long)ns * front);
        need = (need + 3) & ~3ull;
        if (adjoint) {
            rc = ensure_adjoint_front(g, l, std::max(need / 4, 4ull));
        } else if (l > l0) {
            // in the persistent schedule a phase takes a quarter of the next front's quads
            const unsigned long long quads = plain ? need / 4 : std::max(need / 4, 4ull);
            rc = ensure_quads(g, l, quads, g->two_bin);
        }
        if (rc) return rc;
    }
    g->first_ordered = groups > 0 && (plain || l0 == lmax_glob || g->quad[l0 + 1].cap / 4 > 16);
    return ART_OK;
}

// Scheduler state and counters are clear when a trace begins: they are from the start, and the
// last kernel of every trace leaves them so. After a call that failed on the way they are
// cleared here (a clearing that is only captured into a graph leaves them marked as they are).
int begin_trace(art_grid* g)
{
    g->state_dirty_captured = false;
    if (!g->state_clean) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        ART_TRY(cudaMemsetAsync(g->d_state, 0, sizeof(DevState), g->stream));
        ART_TRY(cudaStreamIsCapturing(g->stream, &cs));
        g->state_dirty_captured = cs != cudaStreamCaptureStatusNone;
    }
    g->state_clean = false;
    return ART_OK;
}

// The kernels of a trace are enqueued, the last of which clears the state.
void end_trace(art_grid* g) { g->state_clean = !g->state_dirty_captured; }

// Block size of the trace kernels: the caller's, at most (and by default) what they are built
// for.
int trace_threads(const art_params* p)
{
    return p->block_threads > 0 ? std::min(p->block_threads, kTraceMaxThreads) : kTraceMaxThreads;
}

// Blocks of 256 threads for a pass over n cells, four cells per thread.
int cell_blocks(long long n) { return (int)((n + 1023) / 1024); }

// Opacity per cell length (padded layout) into d_chi, and the two-bin pairs into d_chi2; clears
// the accumulator of a trace with a force (clear4) or without (clear1). Bad densities are flagged in
// st, if given: a pass outside a trace must leave the trace state as it is.
int run_opacity(art_grid* g, const art_params* p, bool two_bin, bool clear4, bool clear1, DevStats* st)
{
    const Coef sH = coef_of(p->sigma_H * g->dx);
    const Coef sd = coef_of(g->nH ? p->sigma_d * g->dx : 0.0);
    k_opacity<<<cell_blocks(g->npad), 256, 0, g->stream>>>(
        g->n[0], g->n[1], g->n[2], g->nH0, g->nH, sH, sd, g->d_chi,
        two_bin ? g->d_chi2 : nullptr, clear4 ? g->d_acc : nullptr,
        clear1 ? reinterpret_cast<float*>(g->d_acc) : nullptr, st);
    ART_TRY(cudaGetLastError());
    return ART_OK;
}

TraceArgs make_args(art_grid* g, const art_params* p, bool adjoint)
{
    const SourceTables& T = g->tables[adjoint ? 1 : 0];
    TraceArgs A;
    std::memset(&A, 0, sizeof(A));
    // the d_max cutoff (read only by the kernels built for a cutoff)
    A.dmax = p->d_max > 0.0 ? to_fix(p->d_max / g->dx, g->fbits) : kNoEnd;
    A.fbits = g->fbits;
    A.unit = (float)std::ldexp(1.0, -g->fbits);
    A.nx = g->n[0];
    A.ny = g->n[1];
    A.nz = g->n[2];
    A.level0 = p->level0;
    A.lmax_glob = g->lmax_glob;
    A.tau_max = (float)p->tau_max;
    A.chi = g->d_chi;
    A.chi2 = g->d_chi2;
    A.srcLn = T.lum;
    A.acc = g->d_acc;
    A.srcL = T.lum;
    A.src = T.src;
    A.levels = g->d_levels + (adjoint ? kNL : 0);
    for (int l = 0; l < kNL; ++l) {
        A.adj[l] = g->adj[l];
        A.quad[l] = g->quad[l];
        if (l > g->lmax_glob) A.adj[l].cap = A.quad[l].cap = 0;
    }
    if (g->first_ordered) A.first = g->d_first;
    A.base_quads = 3u << (2 * p->level0);
    A.nsrc = (unsigned)g->L.size();
    A.npad = (unsigned)g->npad;
    A.sched = g->d_sched;
    A.stats = g->d_stats;
    double ws = p->wait_limit_s == 0.0 ? kDefaultWaitS : p->wait_limit_s;
    A.wait_ns = ws < 0.0 ? -1 : (long long)(ws * 1e9);
    return A;
}

int finish_stats(art_grid* g, art_stats* out)
{
    ART_TRY(cudaStreamSynchronize(g->stream));
    const DevStats& d = *g->h_stats;
    std::memset(out, 0, sizeof(*out));
    out->crossings = d.crossings;
    out->rays_total = d.rays_total;
    for (int l = 0; l < ART_NLEVELS && l < kNL; ++l) out->rays_per_level[l] = d.rays_per_level[l];
    out->destroy = d.destroy;
    out->destroy_expected = g->destroy_expected;
    out->L_in = g->last_L_in;
    out->L_absorbed = g->last_L_in - d.escaped - d.dropped;
    out->L_escaped = d.escaped;
    out->L_dropped = d.dropped;
    out->level_reached = d.level_reached;
    out->level_max = g->last_lmax;
    if (g->last_two_bin) {
        out->Ln_in = g->last_Ln_in;
        out->Ln_escaped = d.escaped_n;
        out->Ln_dropped = d.dropped_n;
        out->Ln_absorbed = g->last_Ln_in - d.escaped_n - d.dropped_n;
    }
    int st = ART_OK;
    if (d.error == -1) st = ART_EINVAL;
    else if (d.error < 0) st = d.error;
    else if (g->last_kind == 0 && d.destroy != g->destroy_expected) st = ART_EACCOUNTING;
    out->status = st;
    return st;
}

}  // namespace art

// ---------------------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------------------
extern "C" {

void art_params_default(art_params* p)
{
    if (!p) return;
    std::memset(p, 0, sizeof(*p));
    p->level0 = 4;
    p->level_max = -1;
    p->m_ray = 4.0;
    p->tau_max = 7.0;
    p->sigma_H = 1.0;
    p->sigma_d = 0.0;
    p->rot[0] = p->rot[4] = p->rot[8] = 1.0;
    p->flags = 0;
    p->schedule = ART_SCHED_PERSISTENT;
}

int art_create_grid(art_grid** out, int nx, int ny, int nz, const double box_lo[3], double dx,
                    const float* d_nH0, const float* d_nH, void* stream)
{
    if (!out) return ART_EINVAL;
    *out = nullptr;
    if (nx <= 0 || ny <= 0 || nz <= 0 || !box_lo || !(dx > 0.0) || !std::isfinite(dx) || !d_nH0)
        return ART_EINVAL;
    for (int a = 0; a < 3; ++a)
        if (!std::isfinite(box_lo[a])) return ART_EINVAL;
    const long long ncell = (long long)nx * ny * nz;
    // the trace kernels index the padded layout (a ring of sentinel cells) in 32 bits
    const long long npad = (long long)(nx + 2) * (ny + 2) * (nz + 2);
    if (npad >= (1ll << 31)) return ART_EINVAL;
    art_grid* g = new (std::nothrow) art_grid();
    if (!g) return ART_ENOMEM;
    g->n[0] = nx; g->n[1] = ny; g->n[2] = nz;
    g->ncell = ncell;
    g->npad = npad;
    for (int a = 0; a < 3; ++a) g->lo[a] = box_lo[a];
    g->dx = dx;
    // as many fraction bits as keep every distance inside the box below 2^61
    g->fbits = 61 - (int)std::ceil(std::log2(
                        std::sqrt((double)nx * nx + (double)ny * ny + (double)nz * nz) + 4.0));
    g->nH0 = d_nH0;
    g->nH = d_nH;
    g->stream = (cudaStream_t)stream;
    int rc = cuda_status(cudaGetDevice(&g->device));
    if (!rc) rc = cuda_status(cudaDeviceGetAttribute(&g->sms, cudaDevAttrMultiProcessorCount, g->device));
    if (!rc) rc = dev_alloc(&g->d_chi, npad + 1);
    g->first_room = (size_t)npad / 32;
    if (!rc) rc = dev_alloc(&g->d_acc, npad + g->first_room);
    if (!rc) rc = dev_alloc(&g->d_levels, 2 * kNL);
    if (!rc) rc = dev_alloc(&g->d_state, 1);
    if (!rc) {
        g->d_sched = &g->d_state->sched;
        g->d_stats = &g->d_state->stats;
        rc = cuda_status(cudaMemsetAsync(g->d_state, 0, sizeof(DevState), g->stream));
        g->state_clean = rc == ART_OK;
    }
    if (!rc) rc = cuda_status(cudaMallocHost((void**)&g->h_stats, sizeof(DevStats)));
    if (rc) {
        art_destroy_grid(g);
        return rc;
    }
    std::memset(g->h_stats, 0, sizeof(DevStats));
    *out = g;
    return ART_OK;
}

int art_update_fields(art_grid* g, const float* d_nH0, const float* d_nH)
{
    if (!g || !d_nH0) return ART_EINVAL;
    g->nH0 = d_nH0;
    g->nH = d_nH;
    return ART_OK;
}

int art_add_sources(art_grid* g, int n, const double* h_pos, const double* h_L)
{
    if (!g || n < 0 || (n > 0 && (!h_pos || !h_L))) return ART_EINVAL;
    for (int s = 0; s < n; ++s) {
        if (!(h_L[s] >= 0.0) || !std::isfinite(h_L[s])) return ART_EINVAL;
        for (int a = 0; a < 3; ++a) {
            double u = (h_pos[3 * s + a] - g->lo[a]) / g->dx;
            if (!(u > 0.0 && u < (double)g->n[a])) return ART_EINVAL;
        }
    }
    g->pos.insert(g->pos.end(), h_pos, h_pos + 3 * (size_t)n);
    g->L.insert(g->L.end(), h_L, h_L + (size_t)n);
    if (g->two_bin) g->Ln.insert(g->Ln.end(), (size_t)n, 0.0);
    return ART_OK;
}

int art_clear_sources(art_grid* g)
{
    if (!g) return ART_EINVAL;
    g->pos.clear();
    g->L.clear();
    g->Ln.clear();
    g->two_bin = false;
    return ART_OK;
}

int art_set_nonionizing(art_grid* g, const double* h_Ln)
{
    if (!g) return ART_EINVAL;
    if (!h_Ln) {
        g->two_bin = false;
        g->Ln.clear();
        return ART_OK;
    }
    if (g->L.empty()) return ART_ESTATE;
    for (size_t s = 0; s < g->L.size(); ++s)
        if (!(h_Ln[s] >= 0.0) || !std::isfinite(h_Ln[s])) return ART_EINVAL;
    g->Ln.assign(h_Ln, h_Ln + g->L.size());
    g->two_bin = true;
    return ART_OK;
}

int art_num_sources(const art_grid* g) { return g ? (int)g->L.size() : 0; }

int art_trace(art_grid* g, const art_params* p, float* d_gamma, float* d_force, float* d_energy,
              art_stats* h_stats)
{
    if (!g || !d_gamma) return ART_EINVAL;
    int rc = check_params(p);
    if (rc) return rc;
    if (g->L.empty()) return ART_ESTATE;
    if ((rc = begin_trace(g))) return rc;
    rc = prepare_trace(g, p, false);
    if (rc) return rc;
    rc = run_opacity(g, p, g->two_bin, d_force != nullptr, d_force == nullptr, g->d_stats);
    if (rc) return rc;
    const int ns = (int)g->L.size();
    const int l0 = p->level0;
    const int threads = trace_threads(p);
    TraceArgs A = make_args(g, p, false);
    if (p->schedule == ART_SCHED_PLAIN) {
        int per_sm = 0;
        const auto kern = level_kernel(g->two_bin, p->d_max > 0.0, d_force != nullptr);
        ART_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0));
        if (per_sm < 1) return ART_EINVAL;
        const int grid = per_sm * g->sms;
        for (int s = 0; s < ns; ++s) {
            k_reset_counts<<<1, 32, 0, g->stream>>>(g->d_sched, (unsigned)(grid * (threads / 32)));
            for (int l = l0; l <= g->src_lmax[s]; ++l)
                kern<<<grid, threads, 0, g->stream>>>(A, l, (unsigned)s);
        }
        if (A.first) {
            const int blocks = std::min((ns + 7) / 8, 16 * g->sms);
            if (d_force) k_add_first<true><<<blocks, 256, 0, g->stream>>>(A);
            else k_add_first<false><<<blocks, 256, 0, g->stream>>>(A);
        }
        ART_TRY(cudaGetLastError());
    } else {
        int per_sm = 0;
        const auto kern = persistent_kernel(g->two_bin, p->d_max > 0.0, d_force != nullptr);
        ART_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0));
        if (per_sm < 1) return ART_EINVAL;
        if (p->blocks_per_sm > 0 && p->blocks_per_sm < per_sm) per_sm = p->blocks_per_sm;
        cudaLaunchConfig_t cfg;
        std::memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3(per_sm * g->sms);
        cfg.blockDim = dim3(threads);
        cfg.stream = g->stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        ART_TRY(cudaLaunchKernelEx(&cfg, kern, A));
    }
    const double dV = g->dx * g->dx * g->dx;
    const float gscale = (float)(p->sigma_H * g->dx / dV);
    const float fscale = (float)(1.0 / dV);
    const float escale = (float)(g->dx / dV);
    const int blocks = cell_blocks(g->ncell);
    if (d_force)
        k_finalize<<<blocks, 256, 0, g->stream>>>(g->n[0], g->n[1], g->n[2], g->d_acc, gscale,
                                                  fscale, escale, d_gamma, d_force, d_energy, g->d_state,
                                                  g->h_stats);
    else
        k_finalize<<<blocks, 256, 0, g->stream>>>(g->n[0], g->n[1], g->n[2],
                                                  reinterpret_cast<const float*>(g->d_acc), gscale,
                                                  fscale, escale, d_gamma, d_force, d_energy, g->d_state,
                                                  g->h_stats);
    ART_TRY(cudaGetLastError());
    end_trace(g);
    double Lin = 0.0;
    for (double v : g->L) Lin += v;
    g->last_L_in = Lin;
    g->last_two_bin = g->two_bin;
    g->last_Ln_in = 0.0;
    for (double v : g->Ln) g->last_Ln_in += v;
    g->last_lmax = g->lmax_glob;
    g->destroy_expected = (unsigned long long)ns * (12ull << (2 * g->lmax_glob));
    g->last_kind = 0;
    g->traced = true;
    if (h_stats) return finish_stats(g, h_stats);
    return ART_OK;
}

int art_get_stats(art_grid* g, art_stats* h_stats)
{
    if (!g || !h_stats) return ART_EINVAL;
    if (!g->traced) return ART_ESTATE;
    return finish_stats(g, h_stats);
}

void art_destroy_grid(art_grid* g)
{
    if (!g) return;
    cudaStreamSynchronize(g->stream);
    dev_free(g->d_chi);
    dev_free(g->d_acc);
    dev_free(g->tables[0].src);
    dev_free(g->tables[1].src);
    free_retired(g);
    dev_free(g->d_levels);
    dev_free(g->d_state);
    dev_free(g->d_rec);
    dev_free(g->d_recf);
    dev_free(g->d_recw);
    dev_free(g->d_chi2);
    for (int l = 0; l < kNL; ++l) {
        dev_free(g->dir[l]);
        dev_free(g->quad[l].rec);
        dev_free(g->quad[l].recn);
        AdjBuf& b = g->adj[l];
        dev_free(b.rec); dev_free(b.parent); dev_free(b.own); dev_free(b.sub);
    }
    if (g->h_stats) cudaFreeHost(g->h_stats);
    delete g;
}

const char* art_strerror(int status)
{
    switch (status) {
    case ART_OK: return "ok";
    case ART_EINVAL: return "invalid argument or input value";
    case ART_ENOMEM: return "out of device or pinned host memory";
    case ART_EQUEUE_OVERFLOW: return "a ray front exceeded its buffer capacity";
    case ART_ETIMEOUT: return "a bounded device-side wait ran out";
    case ART_EACCOUNTING: return "retired-ray weights do not add up to N_src*12*4^l_max";
    case ART_ECUDA: return "CUDA runtime error";
    case ART_ESTATE: return "call out of order (no sources or nothing traced)";
    case ART_EINTERNAL: return "a device-side consistency bound was exceeded";
    default: return "unknown status";
    }
}

}  // extern "C"
