// art_adjoint.cu -- hand-written adjoint of the forward trace for
// loss = sum_c (w_c gamma_c + v_c . force_c) (new; the paper has no adjoint). Gradients with
// respect to log n_H0 per cell and to every source luminosity.
//
// For a segment j of a ray in cell c, with G_j = L_in ds phi(dtau), dL_j = L_in (1 - e^-dtau),
// dtau = chi ds and dtauH = n_H0 sigma_H ds (the part of dtau that scales with n_H0), the
// segment adds w_c k G_j + q_j dL_j to the loss (k converts G to gamma, q_j = (v_c . n)/dV)
// and
//   d loss / d log n_H0[c] += dtauH (w_c k L_in ds phi'(dtau) + q_j L_in e^-dtau - S_after(j)),
// where S_after(j) is the loss of every later segment of the ray and of all of its
// descendants (their entering luminosity carries the factor e^-dtau of segment j). Split
// points and tau_max retirement are held fixed.
//
// Nothing is stored per segment. Rays are traced with unit source luminosity (the loss is
// linear in each L_s; gradients are scaled by L_s when deposited) and every ray is walked twice:
//   pass 1 sums the ray's own weighted segments; a ray that splits stores that sum and its
//     children (a quad with a back-pointer to it);
//   pass 2 (S = own sum + the children's totals) deposits the gradients. The total of a quad's
//     four rays is the parent's sum over its descendants: one writer, no atomics.
// The fronts and the lock-step walks are those of the forward trace (two rays per lane, one in
// small fronts). The persistent schedule takes the deepest unfinished work first: "expand" a
// part of a front (pass 1), then everything below it, then "collapse" that part (pass 2). A warp
// whose 64 rays all end without splitting runs pass 2 at once; such parts (all of the deepest
// fronts, and every part without children) need no collapse.
//
// Before, each lane ran its own state machine of both passes with refills, atomic count-downs of
// the parents and completions in between, with 21 of 32 lanes active. Against that: 9.9 -> 4.6 ms
// on 128^3 / 16 sources with a force term, 1.89 -> 0.70 ms on an odd box with force and dust. What
// bounds it now: without a force term the issue of its instructions (68 % of cycles), with one the
// latency of the 32-byte record gathers first (20 warps per SM hold 40 rays' worth; issue 60 %, and
// the one form of the kernel that spills, 148 bytes).
#include <cmath>
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "art.h"
#include "art_internal.h"

using namespace art;

namespace {


// Running sum in two floats without renormalisation: hi + g is split exactly (two-sum) and
// its rounding error collected in lo.
template <class V>
__device__ __forceinline__ void sum_add(V& hi, V& lo, V g)
{
    const V s = vadd(hi, g);
    const V bb = vsub(s, hi);
    lo = vadd(lo, vadd(vsub(hi, vsub(s, bb)), vsub(g, bb)));
    hi = s;
}

// hi + lo - g for a remainder that only decreases (a >= g >= 0): with |hi| >= g the error of
// hi - g is exact by the fast two-sum; where rounding of earlier steps left hi just below g,
// hi - g is itself exact (Sterbenz) and the error is 0.
template <class V>
__device__ __forceinline__ void sum_take(V& hi, V& lo, V g)
{
    const V s = vsub(hi, g);
    lo = vadd(lo, vsub(vsub(hi, s), g));
    hi = s;
}

// Adds the lanes' parts v of dloss/dL to their sources' FP64 sums: one addition per warp where
// all rays are of one source, as most neighbouring rays of a front are (an addition per ray,
// 11 M to 16 addresses, bound the sweep: 5.77 against 3.85 ms on 128^3 / 16 sources without a
// force term). Warp-uniform; lanes without rays pass v = 0.
__device__ __forceinline__ void dl_add(double* dL, unsigned src, bool valid, double v)
{
    const unsigned lead = __shfl_sync(kFull, src, __ffs(__ballot_sync(kFull, valid)) - 1);
    if (__all_sync(kFull, !valid || src == lead)) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(kFull, v, off);
        if ((threadIdx.x & 31u) == 0 && v != 0.0) atomicAdd(dL + lead, v);
    } else if (valid && v != 0.0) {
        atomicAdd(dL + src, v);
    }
}

// The parts of a cell record: opacity, its neutral-H part, weight, and the force weight of the
// segment q = (v . n) / dV, so that the segment adds q dL to the loss (0 without a force term).
__device__ __forceinline__ float neutral_of(const float4& c) { return c.y; }
__device__ __forceinline__ float neutral_of(const CellF& c) { return c.a.y; }
__device__ __forceinline__ float neutral_of(const CellW& c) { return c.chi; }
__device__ __forceinline__ float weight_of(const float4& c) { return c.z; }
__device__ __forceinline__ float weight_of(const CellF& c) { return c.a.z; }
__device__ __forceinline__ float weight_of(const CellW& c) { return c.w; }
__device__ __forceinline__ float force_weight(const CellF& c, const float* n, float fs)
{
    return fs * fmaf(c.b.x, n[0], fmaf(c.b.y, n[1], c.b.z * n[2]));
}
template <class Cell> struct HasForce { static constexpr bool value = false; };
template <> struct HasForce<CellF> { static constexpr bool value = true; };
template <class Cell> __device__ __forceinline__ const Cell* recs_of(const TraceArgs& A);
template <> __device__ __forceinline__ const float4* recs_of<float4>(const TraceArgs& A) { return A.rec; }
template <> __device__ __forceinline__ const CellF* recs_of<CellF>(const TraceArgs& A) { return A.recf; }
template <> __device__ __forceinline__ const CellW* recs_of<CellW>(const TraceArgs& A) { return A.recw; }

// c = *p if q, as a predicated load.
__device__ __forceinline__ void load_if(bool q, const float4* p, float4& c)
{
    asm("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %5, 0;\n\t"
        "@q ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
        : "+f"(c.x), "+f"(c.y), "+f"(c.z), "+f"(c.w) : "l"(p), "r"((int)q));
}
__device__ __forceinline__ void load_if(bool q, const CellF* p, CellF& c)
{
    asm("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %9, 0;\n\t"
        "@q ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t}"
        : "+f"(c.a.x), "+f"(c.a.y), "+f"(c.a.z), "+f"(c.a.w), "+f"(c.b.x), "+f"(c.b.y),
          "+f"(c.b.z), "+f"(c.b.w)
        : "l"(p), "r"((int)q));
}
__device__ __forceinline__ void load_if(bool q, const CellW* p, CellW& c)
{
    asm("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %3, 0;\n\t"
        "@q ld.global.nc.v2.f32 {%0, %1}, [%2];\n\t}"
        : "+f"(c.chi), "+f"(c.w) : "l"(p), "r"((int)q));
}

// What a lane knows of its quad.
struct QuadInfo {
    unsigned quad, src, pix;  // pix: the lane's first ray
    float L, tau;
    fix rend;
    bool splits;
};

// The rays of a lane during a walk.
template <class Cell, int kWidth>
struct Walkers {
    using V = typename std::conditional<kWidth == 1, float, float2>::type;
    Path W[kWidth];
    Cell cell[kWidth];
    float n[kWidth][3];  // used with a force term only
    V L, tau;
};

template <class Cell, int kWidth>
__device__ __forceinline__ void walkers_start(const TraceArgs& A, const Cell* recs,
                                              const LevelInfo& LV, const QuadInfo& Q, bool valid,
                                              Walkers<Cell, kWidth>& R)
{
    using V = typename Walkers<Cell, kWidth>::V;
    if (valid) {
        const float4 sh = __ldg(&A.src[Q.src].hi);
        const float4 sl = __ldg(&A.src[Q.src].lo);
        const longlong2 xy = __ldg(&A.src[Q.src].xy);
        const longlong2 z_ = __ldg(&A.src[Q.src].z_);
        const df u[3] = {{sh.x, sl.x}, {sh.y, sl.y}, {sh.z, sl.z}};
        const fix ux[3] = {xy.x, xy.y, z_.x};
#pragma unroll
        for (int j = 0; j < kWidth; ++j) {
            df n[3];
            fix code[3];
            load_direction(LV.dir + 3ull * (Q.pix + j), n, code);
            const bool inside = path_start(R.W[j], A.nx, A.ny, A.nz, A.fbits, u, ux, n, code,
                                           LV.r0, LV.r0x);
            // padded cell 0 is a sentinel: a ray that starts outside exits at once
            R.cell[j] = load_cell(recs + (inside ? R.W[j].idx : 0));
#pragma unroll
            for (int a = 0; a < 3; ++a) R.n[j][a] = n[a].hi;
        }
    } else {
#pragma unroll
        for (int j = 0; j < kWidth; ++j) {
            R.W[j] = Path{};
            R.W[j].t[1] = 1ll << 40;
            R.W[j].t[2] = 1ll << 41;
            R.cell[j] = load_cell(recs);
            R.n[j][0] = R.n[j][1] = R.n[j][2] = 0.f;
        }
    }
    R.L = vset<V>(Q.L);
    R.tau = vset<V>(Q.tau);
}

// Walks the lane's rays to their ends. Pass 1 adds each segment's loss w k G + q dL to (hi, lo);
// pass 2 takes it from (hi, lo), what is left of the sum over the segment and all that follows
// it, and deposits the segment's gradient scaled by Ls. Ended rays as in the forward trace.
template <class Cell, int kWidth, int kPass, bool kParts, bool kFirst>
__device__ __forceinline__ void walkers_step(const TraceArgs& A, const Cell* __restrict__ recs,
                                             fix rend, Walkers<Cell, kWidth>& R,
                                             typename Walkers<Cell, kWidth>::V& hi,
                                             typename Walkers<Cell, kWidth>::V& lo, float Ls,
                                             unsigned& ncross)
{
    using V = typename Walkers<Cell, kWidth>::V;
    constexpr bool force = HasForce<Cell>::value;
    V ds, x, wk, hv, q = vset<V>(0.f);
    int key[kWidth];
    bool alive[kWidth], exact = false;
    int high[kWidth];
#pragma unroll
    for (int j = 0; j < kWidth; ++j) {
        bool e;
        alive[j] = !(chi_of(R.cell[j]) < 0.f) & !(vget(R.tau, j) > A.tau_max);
        high[j] = earliest(R.W[j], rend, alive[j], e);
        exact |= e;
        // (a ray that has ended may hold the record of a cell it never entered)
        vget(wk, j) = alive[j] ? weight_of(R.cell[j]) * A.gscale : 0.f;
        vget(hv, j) = neutral_of(R.cell[j]);
        if constexpr (force)
            vget(q, j) = alive[j] ? force_weight(R.cell[j], R.n[j], A.fscale) : 0.f;
    }
    if (exact) {
#pragma unroll
        for (int j = 0; j < kWidth; ++j)
            walk_move<true, kParts>(R.W[j], rend, A.unit, chi_of(R.cell[j]), alive[j], high[j],
                                    -1 - j, (int)A.npad, vget(ds, j), vget(x, j), key[j], ncross);
    } else {
#pragma unroll
        for (int j = 0; j < kWidth; ++j)
            walk_move<false, kParts>(R.W[j], rend, A.unit, chi_of(R.cell[j]), alive[j], high[j],
                                     -1 - j, (int)A.npad, vget(ds, j), vget(x, j), key[j], ncross);
    }
#pragma unroll
    for (int j = 0; j < kWidth; ++j) load_if(alive[j], recs + R.W[j].idx, R.cell[j]);
    V dphi;
    const V ph = phi_dphi<kPass == 2>(x, dphi);
    const V Lin = R.L;
    const V G = vmul(vmul(Lin, ds), ph);
    const V dL = vmul(vmul(Lin, x), ph);
    R.L = vsub(R.L, dL);
    R.tau = vadd(R.tau, x);
    const V g = force ? vfma(q, dL, vmul(wk, G)) : vmul(wk, G);
    if constexpr (kPass == 1) {
        sum_add(hi, lo, g);
    } else {
        sum_take(hi, lo, g);
        const V after = vadd(hi, lo);
        // d(segment loss)/d dtau: w k L_in ds phi' + q L_in e^-dtau (R.L is now L_in e^-dtau)
        V own = vmul(vmul(vmul(wk, Lin), ds), dphi);
        if constexpr (force) own = vfma(q, R.L, own);
        const V val = vmul(vmul(vmul(vset<V>(Ls), hv), ds), vsub(own, after));
        float d[kWidth];
#pragma unroll
        for (int j = 0; j < kWidth; ++j) d[j] = vget(val, j);
        if constexpr (kWidth == 2)
            merge_pair(key[0], d[0], key[1], d[1], -2);
#pragma unroll
        for (int j = 0; j < kWidth; ++j) {
            // the first segments are all in their source's cell: one sum per warp
            if constexpr (kFirst) merge_lanes(key[j], d[j]);
            red_if(A.grad, key[j], d[j]);
        }
    }
}

template <class Cell, int kWidth, int kPass>
__device__ __forceinline__ void walkers_run(const TraceArgs& A, const Cell* __restrict__ recs,
                                            bool base, fix rend, Walkers<Cell, kWidth>& R,
                                            typename Walkers<Cell, kWidth>::V& hi,
                                            typename Walkers<Cell, kWidth>::V& lo, float Ls,
                                            unsigned& ncross)
{
    // the first cells around a source, where a segment can more than double the distance (at
    // most six faces lie within the longest segment, 3^(1/2) cells)
    if (base) {
        walkers_step<Cell, kWidth, kPass, true, true>(A, recs, rend, R, hi, lo, Ls, ncross);
#pragma unroll 1
        for (int k = 1; k < 6; ++k)
            walkers_step<Cell, kWidth, kPass, true, false>(A, recs, rend, R, hi, lo, Ls, ncross);
    }
    for (;;) {
        bool any = false;
#pragma unroll
        for (int j = 0; j < kWidth; ++j)
            any |= !(chi_of(R.cell[j]) < 0.f) & !(vget(R.tau, j) > A.tau_max);
        if (!__any_sync(kFull, any)) break;
#pragma unroll 1
        for (int k = 0; k < kCheckSteps; ++k)
            walkers_step<Cell, kWidth, kPass, false, false>(A, recs, rend, R, hi, lo, Ls, ncross);
    }
}

// One phase on the quads up to `end` of level l, taken 32 lanes at a time from `cursor` (items
// of kWidth rays): expand (pass 1, and pass 2 where no ray of the warp splits) or collapse
// (pass 2 of the quads not done yet). Warp-uniform.
template <class Cell, bool kCut, int kWidth>
__device__ void sweep_front(const TraceArgs& A, int l, bool collapse, unsigned long long* cursor,
                            unsigned long long begin, unsigned long long end)
{
    using V = typename Walkers<Cell, kWidth>::V;
    constexpr unsigned kPerQuad = 4u / kWidth;
    const Cell* const recs = recs_of<Cell>(A);
    const unsigned lane = threadIdx.x & 31u;
    const unsigned lt = (1u << lane) - 1u;
    const LevelInfo& LV = A.levels[l];
    const AdjBuf& B = A.adj[l];
    const bool base = l == A.level0;
    BlockTally& T = block_tally();
    const unsigned items = (unsigned)end * kPerQuad;  // front ends below 2^29 quads
    const unsigned first = (unsigned)begin * kPerQuad;
    Batches batches(cursor, first, items);
    unsigned ncross = 0;

    for (;;) {
        const unsigned b = batches.take(first);
        if (b >= items) break;
        const unsigned item = b + lane;
        bool valid = item < items;
        QuadInfo Q = {item / kPerQuad, 0u, 0u, 0.f, 0.f, kNoEnd, false};
        const unsigned part = item % kPerQuad * kWidth;
        const unsigned ray = 4u * Q.quad + part;  // slot of the lane's first ray
        unsigned parent = 0u;
        if (valid && (collapse || !base)) parent = __ldcg(B.parent + Q.quad);
        if (collapse) valid = valid && parent != kDone;
        if (!__any_sync(kFull, valid)) continue;
        float Ls = 0.f;
        if (valid) {
            if (base) {
                Q.src = Q.quad / A.base_quads;
                Q.pix = 4u * (Q.quad % A.base_quads);
                Q.L = __ldg(&A.src[Q.src].hi).w;
            } else {
                const uint4 r = __ldcg(B.rec + Q.quad);
                Q.src = r.x;
                Q.pix = r.y;
                Q.L = __uint_as_float(r.z);
                Q.tau = __uint_as_float(r.w);
            }
            Q.pix += part;
            Q.splits = l < __float_as_int(__ldg(&A.src[Q.src].lo).w);
            Q.rend = end_radius<kCut>(Q.splits, LV.rmaxx, A.dmax);
            Ls = __ldg(A.srcL + Q.src);
        }

        V hi = vset<V>(0.f), lo = vset<V>(0.f);
        bool second = collapse;  // pass 2 follows
        float total = 0.f;       // loss of the lane's rays and their descendants
        if (!collapse) {
            Walkers<Cell, kWidth> R;
            walkers_start<Cell, kWidth>(A, recs, LV, Q, valid, R);
            walkers_run<Cell, kWidth, 1>(A, recs, base, Q.rend, R, hi, lo, 0.f, ncross);

            // ends: the rays' own sums, and the children of split rays
            bool child[kWidth];
            unsigned nchild = 0, mine = 0, at[kWidth];
            double own = 0.0;
#pragma unroll
            for (int j = 0; j < kWidth; ++j) {
                child[j] = valid && chi_of(R.cell[j]) == kEnded && !(vget(R.tau, j) > A.tau_max) &&
                           splits_at_end<kCut>(Q.splits, LV.rmaxx, A.dmax);
                const unsigned m = __ballot_sync(kFull, child[j]);
                at[j] = __popc(m & lt) + mine;  // children in lane order
                if (j > 0) {
                    at[j] += at[0];
                    at[0] += __popc(m & lt);
                }
                nchild += __popc(m);
                mine += child[j] ? 1u : 0u;
                if (valid) own += (double)vget(hi, j) + (double)vget(lo, j);
            }
            dl_add(A.dL, Q.src, valid, own);
            unsigned slot = 0;
            if (lane == 0) {
                const unsigned nray = kWidth * min(items - b, 32u);
                atomicAdd(&T.rays[l], (unsigned long long)nray);
                atomicAdd(&T.destroy, (unsigned long long)(nray - nchild) * LV.destroy_w);
                if (nchild)
                    slot = (unsigned)atomicAdd(&A.sched->count[l + 1], (unsigned long long)nchild);
            }
            second = nchild == 0;
            if (nchild) {
                const AdjBuf& C = A.adj[l + 1];
                slot = __shfl_sync(kFull, slot, 0);
                if (slot + nchild > C.cap) {
                    atomicCAS(&A.stats->error, 0, -3);  // ART_EQUEUE_OVERFLOW
                } else {
#pragma unroll
                    for (int j = 0; j < kWidth; ++j) {
                        if (child[j]) {
                            __stcg(C.rec + slot + at[j],
                                   make_uint4(Q.src, 4u * (Q.pix + j),
                                              __float_as_uint(0.25f * vget(R.L, j)),
                                              __float_as_uint(vget(R.tau, j))));
                            __stcg(C.parent + slot + at[j], ray + j);
                        }
                    }
                }
                if (valid) {  // kept for the collapse
                    if (base) __stcg(B.parent + Q.quad, 0u);
#pragma unroll
                    for (int j = 0; j < kWidth; ++j) {
                        __stcg(B.own + ray + j, make_float2(vget(hi, j), vget(lo, j)));
                        __stcg(B.sub + ray + j, 0.f);
                    }
                }
            } else if (valid) {
                if (part == 0u) __stcg(B.parent + Q.quad, kDone);
#pragma unroll
                for (int j = 0; j < kWidth; ++j) total += vget(hi, j) + vget(lo, j);
            }
        } else if (valid) {
#pragma unroll
            for (int j = 0; j < kWidth; ++j) {
                const float2 own = __ldcg(B.own + ray + j);
                const df rem = df_add({own.x, own.y}, {__ldcg(B.sub + ray + j), 0.f});
                vget(hi, j) = rem.hi;
                vget(lo, j) = rem.lo;
                total += rem.hi + rem.lo;
            }
        }
        if (second) {
            Walkers<Cell, kWidth> R;
            unsigned again = 0;
            walkers_start<Cell, kWidth>(A, recs, LV, Q, valid, R);
            walkers_run<Cell, kWidth, 2>(A, recs, base, Q.rend, R, hi, lo, Ls, again);
            if (!base) {
#pragma unroll
                for (unsigned off = 1u; off < kPerQuad; off <<= 1)
                    total += __shfl_xor_sync(kFull, total, off);
                if (valid && part == 0u) __stcg(A.adj[l - 1].sub + parent, total);
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ncross += __shfl_down_sync(kFull, ncross, off);
    if (lane == 0 && ncross) atomicAdd(&T.crossings, (unsigned long long)ncross);
}

// Chooses the next phase (run by one thread, all others waiting): the deepest level with open
// quads, which are then collapsed (everything below them is finished), or with quads to expand.
__device__ __forceinline__ void next_sweep(const TraceArgs& A)
{
    Sched* sc = A.sched;
    const int started = __ldcg(&sc->started), kind = __ldcg(&sc->phase_kind);
    const int was = __ldcg(&sc->phase_level);
    int l = -1;
    unsigned long long have = 0, opened = 0, below = 0;
    // the levels are read side by side, from the deepest
#pragma unroll
    for (int k = kLevels - 1; k >= 0; --k) {
        const unsigned long long c = __ldcg(&sc->count[k]);
        unsigned long long open = __ldcg(&sc->open_end[k]);
        // an expanded part without children: every warp ran both passes
        if (started && kind == 0 && k == was && below == 0) open = 0;
        below = c;
        if (l < 0 && (c > 0 || open > 0)) {
            l = k;
            have = c;
            opened = open;
        }
    }
    if (started && kind == 0 && l <= was) sc->open_end[was] = 0;
    if (!started) {
        l = A.level0;
        have = (unsigned long long)A.base_quads * A.nsrc;
    }
    sc->started = 1;
    if (l < 0) {
        sc->done = 1;
        return;
    }
    unsigned long long begin, end;
    if (opened != 0) {
        sc->phase_kind = 1;
        begin = __ldcg(&sc->open_begin[l]);
        end = opened;
        sc->open_end[l] = 0;
    } else {
        sc->phase_kind = 0;
        end = have;
        unsigned long long take = end;
        if (l < A.lmax_glob) take = min(end, A.adj[l + 1].cap / 4);
        if (take == 0) {  // a phase must consume rays, or the schedule never ends
            atomicCAS(&A.stats->error, 0, -8);  // ART_EINTERNAL
            take = end;
        }
        begin = end - take;
        sc->count[l] = begin;
        sc->open_begin[l] = begin;
        sc->open_end[l] = end;
    }
    const int width = front_width(end - begin);
    sc->phase_level = l;
    sc->phase_width = width;
    sc->phase_begin = begin;
    sc->phase_end = end;
    sc->cursor[l] = begin * (unsigned long long)(4 / width) + 32ull * warps_in_grid();
}

template <class Cell, bool kCut>
__global__ void __launch_bounds__(kTraceMaxThreads, kTraceMinBlocks) k_backward_persistent(const __grid_constant__ TraceArgs A)
{
    block_tally_init();
    Sched* sc = A.sched;
    __shared__ int s_level, s_width, s_kind;
    __shared__ unsigned long long s_begin, s_end;
    for (;;) {
        if (!grid_barrier(sc, A.stats, A.wait_ns, [&] { next_sweep(A); })) break;
        if (threadIdx.x == 0) {
            s_level = __ldcg(&sc->done) ? -1 : __ldcg(&sc->phase_level);
            s_width = __ldcg(&sc->phase_width);
            s_kind = __ldcg(&sc->phase_kind);
            s_begin = __ldcg(&sc->phase_begin);
            s_end = __ldcg(&sc->phase_end);
        }
        __syncthreads();
        const int l = s_level;
        if (l < 0) break;
        if (s_width == 2) sweep_front<Cell, kCut, 2>(A, l, s_kind == 1, &sc->cursor[l], s_begin, s_end);
        else sweep_front<Cell, kCut, 1>(A, l, s_kind == 1, &sc->cursor[l], s_begin, s_end);
    }
    block_tally_flush(A.stats);
}

// Per-cell records of the reverse sweep in the padded layout, one gather per crossing, with
// the opacity and its neutral-H part formed exactly as k_opacity forms the forward trace's
// opacity; the sentinel ring and the end marker hold zero weights. The same pass clears the
// gradient and dL and flags bad densities.
struct CellIn {
    float a, b, w, v0, v1, v2;
};
__device__ __forceinline__ void make_record(float4& r, float chi, float h, const CellIn& c)
{
    r = make_float4(chi, h, c.w, 0.f);
}
// with the force weight v
__device__ __forceinline__ void make_record(CellF& r, float chi, float h, const CellIn& c)
{
    r.a = make_float4(chi, h, c.w, 0.f);
    r.b = make_float4(c.v0, c.v1, c.v2, 0.f);
}
// without dust and force term: the neutral-H part is the opacity
__device__ __forceinline__ void make_record(CellW& r, float, float h, const CellIn& c)
{
    r = CellW{h, c.w};
}

template <class Cell>
__global__ void __launch_bounds__(256) k_pack_cells(int nx, int ny, int nz,
                                                    const float* __restrict__ nH0,
                                                    const float* __restrict__ nH, Coef sH, Coef sd,
                                                    const float* __restrict__ w,
                                                    const float* __restrict__ v,
                                                    Cell* __restrict__ rec,
                                                    float* __restrict__ grad,
                                                    double* __restrict__ dL, int nsrc,
                                                    DevStats* __restrict__ st)
{
    if (blockIdx.x == 0)
        for (int s = threadIdx.x; s < nsrc; s += blockDim.x) dL[s] = 0.0;
    const size_t ncell = (size_t)nx * ny * nz;
    bool bad = false;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        make_record(rec[(size_t)(nx + 2) * (ny + 2) * (nz + 2)], kEnded, kEnded, CellIn{});
    each_padded_cell(
        nx, ny, nz,
        [&](unsigned i) {
            CellIn c = {nH0[i], nH ? nH[i] : 0.f, w ? w[i] : 0.f, 0.f, 0.f, 0.f};
            if constexpr (HasForce<Cell>::value) {
                c.v0 = v[i];
                c.v1 = v[ncell + i];
                c.v2 = v[2 * ncell + i];
            }
            return c;
        },
        [&](unsigned q, bool inside, const CellIn& c) {
            float chi = kSentinel, h = kSentinel, dust;
            if (inside) {
                bad = bad || bad_density(c.a) || bad_density(c.b);
                opacities(sH, sd, c.a, c.b, chi, h, dust);
            }
            make_record(rec[q], chi, h, c);
            grad[q] = 0.f;
        });
    if (bad) atomicCAS(&st->error, 0, -1);
}

// Gradient per cell from the padded scratch it was summed in, into the caller's layout.
__global__ void __launch_bounds__(256) k_unpad_grad(int nx, int ny, int nz,
                                                    const float* __restrict__ src,
                                                    float* __restrict__ dst,
                                                    DevState* state, DevStats* host)
{
    finish_state(state, host);
    const unsigned ncell = (unsigned)nx * (unsigned)ny * (unsigned)nz;
    const unsigned long long step = 4ull * gridDim.x * blockDim.x;
    for (unsigned long long base = 4ull * blockIdx.x * blockDim.x + threadIdx.x; base < ncell; base += step) {
        float a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long i = base + (unsigned)k * blockDim.x;
            if (i < ncell) a[k] = __ldcs(src + pad_of((unsigned)i, nx, ny));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long i = base + (unsigned)k * blockDim.x;
            if (i < ncell) dst[i] = a[k];
        }
    }
}

int status_of(cudaError_t e)
{
    if (e == cudaSuccess) return ART_OK;
    return e == cudaErrorMemoryAllocation ? ART_ENOMEM : ART_ECUDA;
}

}  // namespace

extern "C" int art_trace_backward(art_grid* g, const art_params* p, const float* d_w,
                                  const float* d_v, float* d_dlog_nH0, double* d_dL,
                                  art_stats* h_stats)
{
    if (!g || (!d_w && !d_v) || !d_dlog_nH0) return ART_EINVAL;
    int rc = check_params(p);
    if (rc) return rc;
    // the reverse sweep always runs the persistent schedule (all base rays in one buffer)
    art_params pp = *p;
    pp.schedule = ART_SCHED_PERSISTENT;
    p = &pp;
    const int ns = (int)g->L.size();
    if (ns == 0) return ART_ESTATE;
    if (g->two_bin) return ART_EINVAL;  // the reverse sweep covers one-bin traces
    cudaStream_t st = g->stream;
    if ((rc = begin_trace(g))) return rc;
    rc = prepare_trace(g, p, true);
    if (rc) return rc;
    double* dL = d_dL ? d_dL : g->tables[1].dL;
    // the gradient is summed in the padded layout, in the (otherwise idle) accumulator
    float* grad_pad = reinterpret_cast<float*>(g->d_acc);
    const int pack_blocks = cell_blocks(g->npad);
    const int nx = g->n[0], ny = g->n[1], nz = g->n[2];
    const Coef sH = coef_of(p->sigma_H * g->dx);
    const Coef sd = coef_of(g->nH ? p->sigma_d * g->dx : 0.0);
    // without dust the neutral-H opacity is the opacity: an 8-byte record serves
    const bool light = !d_v && sd.full == 0.0;
    if (light) {
        if (!g->d_recw && (rc = status_of(cudaMalloc((void**)&g->d_recw, sizeof(CellW) * (g->npad + 1)))))
            return rc;
        k_pack_cells<CellW><<<pack_blocks, 256, 0, st>>>(nx, ny, nz, g->nH0, g->nH, sH, sd, d_w,
                                                         nullptr, g->d_recw, grad_pad, dL, ns,
                                                         g->d_stats);
    } else if (d_v) {
        if (!g->d_recf && (rc = status_of(cudaMalloc((void**)&g->d_recf, sizeof(CellF) * (g->npad + 1)))))
            return rc;
        k_pack_cells<CellF><<<pack_blocks, 256, 0, st>>>(nx, ny, nz, g->nH0, g->nH, sH, sd, d_w,
                                                         d_v, g->d_recf, grad_pad, dL, ns,
                                                         g->d_stats);
    } else {
        if (!g->d_rec && (rc = status_of(cudaMalloc((void**)&g->d_rec, sizeof(float4) * (g->npad + 1)))))
            return rc;
        k_pack_cells<float4><<<pack_blocks, 256, 0, st>>>(nx, ny, nz, g->nH0, g->nH, sH, sd, d_w,
                                                          nullptr, g->d_rec, grad_pad, dL, ns,
                                                          g->d_stats);
    }
    if ((rc = status_of(cudaGetLastError()))) return rc;
    TraceArgs A = make_args(g, p, true);
    A.rec = g->d_rec;
    A.recf = d_v ? g->d_recf : nullptr;
    A.recw = light ? g->d_recw : nullptr;
    A.grad = grad_pad;
    A.dL = dL;
    const double dV = g->dx * g->dx * g->dx;
    A.gscale = (float)(p->sigma_H * g->dx / dV);
    A.fscale = (float)(1.0 / dV);
    const int threads = trace_threads(p);
    const bool cut = p->d_max > 0.0;
    void (*kern)(TraceArgs) =
        light ? (cut ? k_backward_persistent<CellW, true> : k_backward_persistent<CellW, false>)
        : d_v ? (cut ? k_backward_persistent<CellF, true> : k_backward_persistent<CellF, false>)
              : (cut ? k_backward_persistent<float4, true> : k_backward_persistent<float4, false>);
    int per_sm = 0;
    if ((rc = status_of(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0))))
        return rc;
    if (per_sm < 1) return ART_EINVAL;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(per_sm * g->sms);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if ((rc = status_of(cudaLaunchKernelEx(&cfg, kern, A)))) return rc;
    k_unpad_grad<<<cell_blocks(g->ncell), 256, 0, st>>>(nx, ny, nz, grad_pad, d_dlog_nH0,
                                                       g->d_state, g->h_stats);
    if ((rc = status_of(cudaGetLastError()))) return rc;
    end_trace(g);
    g->last_L_in = 0.0;
    for (double v : g->L) g->last_L_in += v;
    g->last_lmax = g->lmax_glob;
    g->destroy_expected = (unsigned long long)ns * (12ull << (2 * g->lmax_glob));
    g->last_kind = 1;
    g->traced = true;
    if (h_stats) return finish_stats(g, h_stats);
    return ART_OK;
}
