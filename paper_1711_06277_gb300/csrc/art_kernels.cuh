// art_kernels.cuh -- forward trace kernels of the GB300 adaptive ray trace.
//
// Work decomposition. The rays of one HEALPix level form a "front" of quads, the four
// children of a split ray, in the order their parents ended. A warp takes 64 neighbouring rays
// at a time, two per lane, and walks them in lock step from their start radius to their ends
// (Sec. 2.1: r_max(l), tau > tau_max or the grid boundary), then appends the children of its
// split rays to the next front with one reservation. Small fronts are walked one ray per lane.
//
// What bounds it: the SM's reductions and its instruction issue, about equally. An SM issues a
// 16-byte reduction at 1.36 clocks per lane when the lanes hit different sectors (44 clocks per
// full warp, measured), and equal addresses within a warp are not combined: one reduction per
// ray and step capped the trace at 2.2e11 crossings per second, whatever the instruction
// count. Two siblings lie in the same cell in 44 % of their steps (m_ray = 4), and merging them
// within a thread costs a compare and four predicated adds, where merging across lanes costs
// shuffles. Lock step keeps siblings together and needs no refill of idle lanes: neighbouring
// rays of a front take nearly the same number of steps (88-93 % lane use over a warp). Four rays
// per lane merge more (0.51 against 0.68 sectors per crossing) but leave 12 instead of 20 warps
// per SM (16.7 against 14.3 ms on 256^3 / 16 sources, before the step was trimmed further).
// Against one ray per lane with refills (and floating-point pairs for the distances):
// 85.5 -> 51.6 ms on 256^3 / 64 sources, 619 -> 409 ms on 512^3 / 64 sources, 3.55 -> 0.28 ms on
// 128^3 / 64 sources cut at 19 cells, where rays of 7 steps had waited for refills every 64.
//
// Two schedules share that routine:
//   * plain: one launch per (source, level), fronts kept whole;
//   * persistent: one cooperative launch for all sources. The launch loops over phases;
//     each phase consumes the top part of the deepest non-empty front, at most a quarter of
//     the next front's capacity, so the children always fit. Deepest-first order keeps every
//     buffer bounded, which is the memory role the paper's last-in-first-out ray stack plays
//     (Sec. 2.2). A grid barrier with a bounded wait separates phases; the last block to
//     arrive chooses the next phase. The retired-ray weights 4^(l_max - l) are summed as the
//     paper's destroy counter (Sec. 2.2).
#pragma once

#include <type_traits>

#include "art_device.cuh"

namespace art {

// ---------------------------------------------------------------------------------------
// HEALPix nested directions in FP64 (Gorski et al. 2005), rotated, split into hi + lo
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t even_bits(uint64_t x)
{
    x &= 0x5555555555555555ull;
    x = (x | (x >> 1)) & 0x3333333333333333ull;
    x = (x | (x >> 2)) & 0x0f0f0f0f0f0f0f0full;
    x = (x | (x >> 4)) & 0x00ff00ff00ff00ffull;
    x = (x | (x >> 8)) & 0x0000ffff0000ffffull;
    x = (x | (x >> 16)) & 0x00000000ffffffffull;
    return (uint32_t)x;
}

// cos and sin of pi * num / den (den > 0), exact at multiples of 1/2, cos = sin at 1/4.
__device__ __forceinline__ void cossin_pi_frac(long long num, long long den, double& c, double& s)
{
    long long m = num % (2 * den);
    if (m < 0) m += 2 * den;
    double sgn_c = 1.0, sgn_s = 1.0;
    if (m >= den) { m -= den; sgn_c = -1.0; sgn_s = -1.0; }  // shift by pi
    if (2 * m > den) { m = den - m; sgn_c = -sgn_c; }        // reflect about pi/2
    double cv, sv;
    if (m == 0) { cv = 1.0; sv = 0.0; }
    else if (2 * m == den) { cv = 0.0; sv = 1.0; }
    else if (4 * m == den) { cv = 0.70710678118654752440; sv = cv; }
    else sincospi((double)m / (double)den, &sv, &cv);
    c = sgn_c * cv;
    s = sgn_s * sv;
}

__global__ void k_directions(int level, unsigned long long npix, double r0, double r1, double r2,
                             double r3, double r4, double r5, double r6, double r7, double r8,
                             int rotate, double fscale, float4* __restrict__ dir)
{
    unsigned long long p = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    if (p >= npix) return;
    const long long ns = 1ll << level;
    const unsigned long long nface = (unsigned long long)(ns * ns);
    const int face = (int)(p / nface);
    const unsigned long long q = p - (unsigned long long)face * nface;
    const long long x = even_bits(q), y = even_bits(q >> 1);
    const int row = face >> 2;                      // 0 north, 1 equator, 2 south
    const long long ring = (long long)(row + 2) * ns - x - y - 1;
    long long nr;
    int shift = 0;
    double z, st;
    if (ring < ns || ring > 3 * ns) {
        nr = ring < ns ? ring : 4 * ns - ring;
        double a = (double)(nr * nr) / (3.0 * (double)(ns * ns));
        z = ring < ns ? 1.0 - a : a - 1.0;
        st = sqrt(a * (2.0 - a));
    } else {
        nr = ns;
        shift = (int)((ring - ns) & 1);
        z = (double)(4 * ns - 2 * ring) / (3.0 * (double)ns);
        st = sqrt((1.0 - z) * (1.0 + z));
    }
    const int col = (row == 1) ? 2 * (face & 3) : 2 * (face & 3) + 1;
    long long jp = (col * nr + x - y + 1 + shift) / 2;
    if (jp > 4 * nr) jp -= 4 * nr;
    if (jp < 1) jp += 4 * nr;
    double c, s;
    cossin_pi_frac(2 * jp - shift - 1, 4 * nr, c, s);
    double v[3] = {st * c, st * s, z};
    double w[3];
    if (rotate) {
        w[0] = r0 * v[0] + r1 * v[1] + r2 * v[2];
        w[1] = r3 * v[0] + r4 * v[1] + r5 * v[2];
        w[2] = r6 * v[0] + r7 * v[1] + r8 * v[2];
    } else {
        w[0] = v[0]; w[1] = v[1]; w[2] = v[2];
    }
    // Distances along directions of length 1/2 or more stay below kFar inside the box, and every
    // step of a walk moves its ray. Where a matrix that is no rotation makes them shorter, they
    // are lengthened to 1: a ray whose faces all lie beyond kFar would never end.
    const double len2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    if (!(len2 >= 0.25)) {
        const double scale = len2 > 0.0 ? 1.0 / sqrt(len2) : 0.0;
        for (int a = 0; a < 3; ++a) w[a] = scale > 0.0 ? w[a] * scale : (a == 0 ? 1.0 : 0.0);
    }
    float h[3], l[3];
    fix d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (fabs(w[a]) < 5.9604644775390625e-08) w[a] = 0.0;  // 2^-24
        h[a] = __double2float_rn(w[a]);
        l[a] = __double2float_rn(w[a] - (double)h[a]);
        // distance between faces, 1/|n_a| (fixed-point, fscale = 2^fbits)
        d[a] = w[a] != 0.0 ? encode_spacing(fscale / fabs(w[a])) : 0;
    }
    // layout: {n_hx, n_hy, n_hz, n_lx}, {n_ly, n_lz, d_x}, {d_y, d_z}
    dir[3 * p] = make_float4(h[0], h[1], h[2], l[0]);
    dir[3 * p + 1] = make_float4(l[1], l[2], __uint_as_float((unsigned)d[0]),
                                 __uint_as_float((unsigned)(d[0] >> 32)));
    *reinterpret_cast<longlong2*>(dir + 3 * p + 2) = make_longlong2(d[1], d[2]);
}

// chi per cell length (dx) in FP32 from the density fields, in the padded layout with the
// sentinel ring; flags bad densities in st (if given) and clears the accumulator (acc4 with force,
// acc1 without).
__global__ void __launch_bounds__(256) k_opacity(int nx, int ny, int nz,
                                                 const float* __restrict__ nH0,
                                                 const float* __restrict__ nH, Coef sH, Coef sd,
                                                 float* __restrict__ chi,
                                                 float2* __restrict__ chi2,
                                                 float4* __restrict__ acc4,
                                                 float* __restrict__ acc1,
                                                 DevStats* __restrict__ st)
{
    bool bad = false;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const size_t npad = (size_t)(nx + 2) * (ny + 2) * (nz + 2);
        chi[npad] = kEnded;
        if (chi2) chi2[npad] = make_float2(kEnded, 0.f);
    }
    each_padded_cell(
        nx, ny, nz, [&](unsigned i) { return make_float2(nH0[i], nH ? nH[i] : 0.f); },
        [&](unsigned q, bool inside, float2 v) {
            float c = kSentinel, h, dust = 0.f;
            if (inside) {
                bad = bad || bad_density(v.x) || bad_density(v.y);
                opacities(sH, sd, v.x, v.y, c, h, dust);
            }
            chi[q] = c;
            if (chi2) chi2[q] = make_float2(c, dust);
            if (acc4) acc4[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (acc1) acc1[q] = 0.f;
        });
    if (bad && st) atomicCAS(&st->error, 0, -1);
}

// The per-cell records a trace gathers: opacities (one bin) or opacity pairs (two bins).
template <class Cell> __device__ __forceinline__ const Cell* cells_of(const TraceArgs& A);
template <> __device__ __forceinline__ const float* cells_of<float>(const TraceArgs& A) { return A.chi; }
template <> __device__ __forceinline__ const float2* cells_of<float2>(const TraceArgs& A) { return A.chi2; }

__device__ __forceinline__ void load_pair(const float* p, float& a, float& b) { a = __ldg(p); b = 0.f; }
__device__ __forceinline__ void load_pair(const float2* p, float& a, float& b)
{
    const float2 v = __ldg(p);
    a = v.x;
    b = v.y;
}

// Photons of the rays of a lane, side by side (V: float or float2).
template <class V>
struct Photons {
    V L, tau;
    V Lc;        // photon ledger: the rounding error of this walk's L updates; tallied with
                 // the ray, never used for deposits
    V n[3];      // directions (hi parts) for momentum deposits
    V Ln, taun, Lnc;  // non-ionizing bin (two-bin traces only)
};

// L - dL, and its rounding error (Fast2Sum, dL <= L) for the photon ledger: where a cell is
// nearly transparent dL falls below half an ulp of L, so the deposited dL never leaves L. The
// deposits keep using L itself, whose relative accuracy survives strong attenuation (L + Lc
// carries the absolute error of all deposits instead); only the tallies of retired rays take
// L + Lc.
template <class V>
__device__ __forceinline__ void lose(V& L, V& Lc, V dL)
{
    const V Lnew = vsub(L, dL);
    Lc = vadd(Lc, vsub(vsub(L, Lnew), dL));
    L = Lnew;
}

// What a segment adds to its cell: (sum L ds phi, sum dL n), or the first alone in traces
// without a force, whose accumulator is a quarter as large and holds eight cells per sector
// instead of two.
template <bool kForce> struct DepositOf { using type = float4; };
template <> struct DepositOf<false> { using type = float; };
template <bool kForce>
__device__ __forceinline__ typename DepositOf<kForce>::type* accumulator(const TraceArgs& A)
{
    return reinterpret_cast<typename DepositOf<kForce>::type*>(A.acc);
}

// The first segments of base rays lie in their source's cell, or in the up to eight cells around
// it where it sits on a face, an edge or a corner. The sum of each group of 32 rays and cell is
// kept until the base front is done, and one warp per source then adds them up, so that the rate
// next to a single source, the largest of the field, and with it the substep size are the same in
// every run; added as the warps got to them, 96 sums at l0 = 4 differed by 1e-7 to 6e-7 from run to
// run. They are added in two floats: their order in one float leaves up to 8e-7 (equal sums of
// symmetric directions in a row are rounded alike). The 6 and 24 sums of l0 = 2 and 3 are added in
// one, where the former walk (64 base rays per warp, the first half of each first) came to one
// value in nearly every run, and in the order that gives it most often: the last groups first, those
// of odd number at l0 = 3 one place late.
template <class D>
struct FirstSegments {  // of the rays of a block on their way
    D value[2][kTraceMaxThreads];
    int key[2][kTraceMaxThreads];
};
template <class D>
__device__ __forceinline__ FirstSegments<D>& first_segments()
{
    __shared__ FirstSegments<D> f;
    return f;
}
template <class D>
__device__ __forceinline__ D* first_sums(const TraceArgs& A)
{
    return reinterpret_cast<D*>(A.first);
}

// Keeps the sums of one group at `to`, one per cell (bit a of a cell's number says that it is the
// lower of the two on axis a). A lane's ray lies `below` cells of the padded layout below the
// source's cell, if it has a segment at all (some). Warp-uniform.
template <class D>
__device__ __forceinline__ void keep_first(D* to, int sy, int sz, int below, bool some, D v)
{
    const unsigned lane = threadIdx.x & 31u;
    int o = 0;
    if (below >= sz) { o |= 4; below -= sz; }
    if (below >= sy) { o |= 2; below -= sy; }
    o |= below;
    D mine{};  // lane o keeps the sum of cell o
    unsigned left = __ballot_sync(kFull, some);
    while (left) {
        const int cell = __shfl_sync(kFull, o, __ffs(left) - 1);
        const bool in = some && o == cell;
        D sum = in ? v : D{};
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) add_to(sum, shifted(sum, off));  // lane 0's is whole
        sum = from_lane(sum, 0);
        if ((int)lane == cell) mine = sum;
        left &= ~__ballot_sync(kFull, in);
    }
    if (lane < 8u) __stcg(to + lane, mine);
}

// The sum of a source's kept sums for cell `lane % 8`, in every lane; `from` are its first group's.
// Four groups side by side. Warp-uniform.
template <class D>
__device__ __forceinline__ D sum_first(const D* from, unsigned groups)
{
    const unsigned lane = threadIdx.x & 31u;
    from += lane % 8u;
    D sum{}, rest{};
    if (groups <= 24u) {
        const int last = (int)groups / 2 - 1, late = groups > 6u ? 1 : 0;
#pragma unroll 6
        for (int t = 0; t < (int)groups; ++t) {
            // even groups from the last down, each followed by the odd one of its pair (l0 = 2) or
            // of the pair before; at l0 = 3 the last even one begins and the first odd one ends
            const int u = t - late, odd = u & 1;
            const int i = odd ? last - (u >> 1) : last - late - (u >> 1);
            add_to(sum, __ldcg(from + 8 * (u < 0 ? 2 * last : i < 0 ? 1 : 2 * i + odd)));
        }
        return sum;
    }
    for (unsigned t = lane / 8u; t < groups; t += 32u) {
        D v[8];  // eight loads in flight
#pragma unroll
        for (unsigned k = 0; k < 8u; ++k) v[k] = t + 4u * k < groups ? __ldcg(from + 8u * (t + 4u * k)) : D{};
#pragma unroll
        for (unsigned k = 0; k < 8u; ++k) add_pair(sum, rest, v[k]);
    }
#pragma unroll
    for (int off = 8; off < 32; off <<= 1) {
        const D s2 = across(sum, off), r2 = across(rest, off);
        add_pair(sum, rest, s2);
        add_to(rest, r2);
    }
    return with_rest(sum, rest);
}

// Adds the kept sums of all sources to the accumulator, a warp per source, the warps with the last
// batches, if any, of a front first. In the persistent schedule every warp gets here after its share
// of the front that follows the base, while others still walk; as a function apart, and called
// after the walk, it costs nothing measurable (in line or before the walk 2 to 3 %, by the walk's
// registers; as a kernel of its own 7 us; in the last kernel, by the blocks of the sources' cells, 7 us
// with one source and 46 us with 64).
template <class D>
__device__ __noinline__ void add_first(const TraceArgs& A, D* acc)
{
    const unsigned o = threadIdx.x % 8u;  // the lane's cell
    const unsigned groups = A.base_quads / 8u;
    for (unsigned s = warps_in_grid() - 1u - warp_in_grid(); s < A.nsrc; s += warps_in_grid()) {
        const D sum = sum_first(first_sums<D>(A) + 8ull * groups * s, groups);
        if (threadIdx.x % 32u < 8u && !is_zero(sum))
            red_if(acc, source_cell(A.src[s]) - (int)(o & 1u) -
                            (A.nx + 2) * ((int)(o >> 1 & 1u) + (A.ny + 2) * (int)(o >> 2)), sum);
    }
}

// Walks kWidth (1 or 2) rays per lane: the rays of quads [begin, end) of level l, taken 32
// lanes at a time from `cursor`, which counts items of kWidth rays. Base-level quads are
// implied by their index (src0 is the first source), deeper ones are records. strided says that
// base rays come in whole groups of 64: where a lane takes two, they are 32 apart instead of
// neighbours, so that a group of 32 is the same at both widths. Warp-uniform.
template <class Cell, bool kCut, bool kForce, int kWidth>
__device__ void walk_front(const TraceArgs& A, const Cell* __restrict__ cells, int l,
                           unsigned long long* cursor, unsigned long long begin,
                           unsigned long long end, unsigned src0, bool strided)
{
    constexpr bool two = TwoBin<Cell>::value;
    using V = typename std::conditional<kWidth == 1, float, float2>::type;
    constexpr unsigned kPerQuad = 4u / kWidth;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned lt = (1u << lane) - 1u;
    const LevelInfo& LV = A.levels[l];
    const bool base = l == A.level0;
    BlockTally& T = block_tally();
    using D = typename DepositOf<kForce>::type;
    D* const acc = accumulator<kForce>(A);
    FirstSegments<D>& F = first_segments<D>();
    const unsigned items = (unsigned)end * kPerQuad;  // front ends below 2^29 quads
    const unsigned first = (unsigned)begin * kPerQuad;
    Batches batches(cursor, first, items);
    unsigned ncross = 0;

    for (;;) {
        const unsigned b = batches.take(first);
        if (b >= items) break;

        // ---- set-up: a part of a quad per lane
        const unsigned item = b + lane;
        const bool valid = item < items;
        Path W[kWidth];
        Photons<V> P;
        float cell[kWidth], celln[kWidth];
        unsigned s = 0, pix = 0;
        const unsigned apart = kWidth == 2 && strided ? 32u : 1u;  // between a lane's pixels
        fix rend = kNoEnd;
        bool splits = false;
        P.L = P.tau = P.Lc = P.Ln = P.taun = P.Lnc = vset<V>(0.f);
        if (valid) {
            unsigned quad = item / kPerQuad, part = item % kPerQuad * kWidth;
            if (kWidth == 2 && strided) {
                quad = (2u * b + lane) / 4u;
                part = lane % 4u;
            }
            float L0 = 0.f, tau0 = 0.f, Ln0 = 0.f, taun0 = 0.f;
            if (base) {
                s = src0 + quad / A.base_quads;
                pix = 4u * (quad % A.base_quads);
            } else {
                const uint4 r = __ldcg(A.quad[l].rec + quad);
                s = r.x;
                pix = r.y;
                L0 = __uint_as_float(r.z);
                tau0 = __uint_as_float(r.w);
                if constexpr (two) {
                    const float2 rn = __ldcg(A.quad[l].recn + quad);
                    Ln0 = rn.x;
                    taun0 = rn.y;
                }
            }
            pix += part;
            const float4 sh = __ldg(&A.src[s].hi);
            const float4 sl = __ldg(&A.src[s].lo);
            const longlong2 xy = __ldg(&A.src[s].xy);
            const longlong2 z_ = __ldg(&A.src[s].z_);
            const df u[3] = {{sh.x, sl.x}, {sh.y, sl.y}, {sh.z, sl.z}};
            const fix ux[3] = {xy.x, xy.y, z_.x};
            splits = l < __float_as_int(sl.w);
            rend = end_radius<kCut>(splits, LV.rmaxx, A.dmax);
            if (base) {
                L0 = sh.w;
                if constexpr (two) Ln0 = __ldg(A.srcLn + s);
            }
#pragma unroll
            for (int j = 0; j < kWidth; ++j) {
                df n[3];
                fix code[3];
                load_direction(LV.dir + 3ull * (pix + j * apart), n, code);
                const bool inside = path_start(W[j], A.nx, A.ny, A.nz, A.fbits, u, ux, n, code,
                                               LV.r0, LV.r0x);
                // padded cell 0 is a sentinel: a ray that starts outside exits at once
                load_pair(cells + (inside ? W[j].idx : 0), cell[j], celln[j]);
#pragma unroll
                for (int a = 0; a < 3; ++a) vget(P.n[a], j) = n[a].hi;
            }
            P.L = vset<V>(L0);
            P.tau = vset<V>(tau0);
            P.Ln = vset<V>(Ln0);
            P.taun = vset<V>(taun0);
        } else {
#pragma unroll
            for (int j = 0; j < kWidth; ++j) {
                W[j] = Path{};
                W[j].t[1] = 1ll << 40;
                W[j].t[2] = 1ll << 41;
                cell[j] = kSentinel;
                celln[j] = 0.f;
            }
            P.n[0] = P.n[1] = P.n[2] = vset<V>(0.f);
        }

        // ---- walk: a ray that has ended sits in a cell of negative opacity (the sentinel
        // ring where it left the grid, the end marker where it reached its end radius) or has
        // passed tau_max, and does nothing more. In two-bin traces the packet is used up once
        // its dust-only depth (never the larger one) passes tau_max.
        auto step = [&](auto first) {
            int key[kWidth];
            V ds, x, xn = vset<V>(0.f);
            bool alive[kWidth], exact = false;
            int high[kWidth];
#pragma unroll
            for (int j = 0; j < kWidth; ++j) {
                bool e;
                alive[j] = !(cell[j] < 0.f) & !(vget(two ? P.taun : P.tau, j) > A.tau_max);
                high[j] = earliest(W[j], rend, alive[j], e);
                exact |= e;
            }
            if (exact) {
#pragma unroll
                for (int j = 0; j < kWidth; ++j)
                    walk_move_load<true>(W[j], rend, A.unit, cell[j], alive[j], high[j], -1 - j,
                                         (int)A.npad, cells, vget(ds, j), vget(x, j), key[j],
                                         ncross);
            } else {
#pragma unroll
                for (int j = 0; j < kWidth; ++j)
                    walk_move_load<false>(W[j], rend, A.unit, cell[j], alive[j], high[j], -1 - j,
                                          (int)A.npad, cells, vget(ds, j), vget(x, j), key[j],
                                          ncross);
            }
            if constexpr (two) {
#pragma unroll
                for (int j = 0; j < kWidth; ++j) {
                    vget(xn, j) = celln[j] * vget(ds, j);
                    if (alive[j]) celln[j] = __ldg(&cells[W[j].idx].y);
                }
            }
            // deposit and loss
            P.tau = vadd(P.tau, x);
            const V ph = phi_of(x);
            const V Lds = vmul(P.L, ds);
            const V dL = vmul(vmul(P.L, x), ph);
            lose(P.L, P.Lc, dL);
            [[maybe_unused]] V dm = dL;  // momentum of both bins
            if constexpr (two) {
                P.taun = vadd(P.taun, xn);
                const V dLn = vmul(vmul(P.Ln, xn), phi_of(xn));
                lose(P.Ln, P.Lnc, dLn);
                dm = vadd(dm, dLn);
            }
            // (the parts of a reduction need registers in a row: formed one by one, they need no
            // moves out of the pairs of two rays, 3 % of the trace)
            D v[kWidth];
#pragma unroll
            for (int j = 0; j < kWidth; ++j) {
                const float G = __fmul_rn(vget(Lds, j), vget(ph, j));
                if constexpr (kForce)
                    v[j] = make_float4(G, __fmul_rn(vget(dm, j), vget(P.n[0], j)),
                                       __fmul_rn(vget(dm, j), vget(P.n[1], j)),
                                       __fmul_rn(vget(dm, j), vget(P.n[2], j)));
                else
                    v[j] = G;
            }
            if constexpr (decltype(first)::value) {
#pragma unroll
                for (int j = 0; j < kWidth; ++j) {
                    F.value[j][threadIdx.x] = v[j];
                    F.key[j][threadIdx.x] = key[j];
                }
            } else {
                if constexpr (kWidth == 2) merge_pair(key[0], v[0], key[1], v[1], -2);
#pragma unroll
                for (int j = 0; j < kWidth; ++j) red_if(acc, key[j], v[j]);
            }
        };
        if (base) step(std::true_type{});
        for (;;) {
            bool any = false;
#pragma unroll
            for (int j = 0; j < kWidth; ++j)
                any |= !(cell[j] < 0.f) & !(vget(two ? P.taun : P.tau, j) > A.tau_max);
            if (!__any_sync(kFull, any)) break;
#pragma unroll 1
            for (int k = 0; k < kCheckSteps; ++k) step(std::false_type{});
        }

        // ---- first segments of base rays (here, where the walk's registers are free)
        if (base) {
            D v[kWidth];
            int key[kWidth];
#pragma unroll
            for (int j = 0; j < kWidth; ++j) {
                v[j] = F.value[j][threadIdx.x];
                key[j] = F.key[j][threadIdx.x];
            }
            if (strided && A.first) {
                const int at = source_cell(A.src[s]);
                D* const to = first_sums<D>(A) + 8u * (src0 * (A.base_quads / 8u) + kWidth * b / 32u);
#pragma unroll
                for (int j = 0; j < kWidth; ++j)
                    keep_first(to + 8 * j, A.nx + 2, (A.nx + 2) * (A.ny + 2), at - key[j], key[j] >= 0, v[j]);
            } else {
                if constexpr (kWidth == 2)
                    if (!strided) merge_pair(key[0], v[0], key[1], v[1], -2);
#pragma unroll
                for (int j = 0; j < kWidth; ++j) {
                    merge_lanes(key[j], v[j]);
                    red_if(acc, key[j], v[j]);
                }
            }
        }

        // ---- ends: the children of split rays, and tallies (while the reservation of the
        // children's slots is on its way)
        bool child[kWidth], drop[kWidth];
        unsigned nchild = 0, mine = 0, at[kWidth];
#pragma unroll
        for (int j = 0; j < kWidth; ++j) {
            drop[j] = vget(two ? P.taun : P.tau, j) > A.tau_max;
            child[j] = valid && cell[j] == kEnded && !drop[j] &&
                       splits_at_end<kCut>(splits, LV.rmaxx, A.dmax);
            const unsigned m = __ballot_sync(kFull, child[j]);
            // children in pixel order: group after group, or lane after lane
            at[j] = __popc(m & lt) + (apart > 1u ? nchild : mine);
            if (apart == 1u && j > 0) {
                at[j] += at[0];
                at[0] += __popc(m & lt);
            }
            nchild += __popc(m);
            mine += child[j] ? 1u : 0u;
        }
        unsigned slot = 0;
        if (lane == 0 && nchild)
            slot = (unsigned)atomicAdd(&A.sched->count[l + 1], (unsigned long long)nchild);
        df esc = {0.f, 0.f}, dropped = {0.f, 0.f}, escn = {0.f, 0.f}, droppedn = {0.f, 0.f};
        if (valid) {
            // leaving the box or cut at d_max: escaped; tau > tau_max: dropped. A split ray
            // leaves its ledger residual: its children start from L itself.
#pragma unroll
            for (int j = 0; j < kWidth; ++j) {
                df& to = drop[j] ? dropped : esc;
                df_accumulate(to, child[j] ? 0.f : vget(P.L, j));
                df_accumulate(to, vget(P.Lc, j));
                if constexpr (two) {
                    df& ton = drop[j] ? droppedn : escn;
                    df_accumulate(ton, child[j] ? 0.f : vget(P.Ln, j));
                    df_accumulate(ton, vget(P.Lnc, j));
                }
            }
        }
        T.escaped[threadIdx.x] += (double)esc.hi + (double)esc.lo;
        if (dropped.hi != 0.f) T.dropped[threadIdx.x] += (double)dropped.hi + (double)dropped.lo;
        if constexpr (two) {
            T.escaped_n[threadIdx.x] += (double)escn.hi + (double)escn.lo;
            T.dropped_n[threadIdx.x] += (double)droppedn.hi + (double)droppedn.lo;
        }
        if (lane == 0) {
            const unsigned nray = kWidth * min(items - b, 32u);
            atomicAdd(&T.rays[l], (unsigned long long)nray);
            atomicAdd(&T.destroy, (unsigned long long)(nray - nchild) * LV.destroy_w);
        }
        if (nchild) {
            const QuadBuf& C = A.quad[l + 1];
            slot = __shfl_sync(kFull, slot, 0);
            // every slot below the capacity is written, whatever a front leaves out: the next
            // launch of the plain schedule reads them all
            const unsigned cap = (unsigned)C.cap, room = slot < cap ? min(nchild, cap - slot) : 0u;
            if (room < nchild) atomicCAS(&A.stats->error, 0, -3);  // ART_EQUEUE_OVERFLOW
#pragma unroll
            for (int j = 0; j < kWidth; ++j) {
                if (child[j] && at[j] < room) {
                    __stcg(C.rec + slot + at[j],
                           make_uint4(s, 4u * (pix + j * apart),
                                      __float_as_uint(0.25f * vget(P.L, j)),
                                      __float_as_uint(vget(P.tau, j))));
                    if constexpr (two)
                        __stcg(C.recn + slot + at[j],
                               make_float2(0.25f * vget(P.Ln, j), vget(P.taun, j)));
                }
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ncross += __shfl_down_sync(kFull, ncross, off);
    if (lane == 0 && ncross) atomicAdd(&T.crossings, (unsigned long long)ncross);
}

// Base rays are taken 32 apart where the front's quads [begin, end) are whole groups of 64 rays
// of one source.
__device__ __forceinline__ bool front_strided(const TraceArgs& A, bool base,
                                              unsigned long long begin, unsigned long long end)
{
    return base && A.base_quads % 16u == 0u && begin % 16u == 0u && end % 16u == 0u;
}

template <class Cell, bool kCut, bool kForce>
__device__ __forceinline__ void run_front(const TraceArgs& A, int l, int width,
                                          unsigned long long* cursor, unsigned long long begin,
                                          unsigned long long end, unsigned src0, bool strided)
{
    if (width == 2) walk_front<Cell, kCut, kForce, 2>(A, cells_of<Cell>(A), l, cursor, begin, end, src0, strided);
    else walk_front<Cell, kCut, kForce, 1>(A, cells_of<Cell>(A), l, cursor, begin, end, src0, strided);
}

// Plain schedule: the whole front of level l of source s.
template <class Cell, bool kCut, bool kForce>
__global__ void __launch_bounds__(kTraceMaxThreads, kTraceMinBlocks) k_trace_level(const __grid_constant__ TraceArgs A, int l, unsigned s)
{
    block_tally_init();
    // a front that overflowed (status set by the writer) is cut at the buffer capacity
    const unsigned long long end =
        l == A.level0 ? (unsigned long long)A.base_quads
                      : min(*((volatile unsigned long long*)&A.sched->count[l]), A.quad[l].cap);
    run_front<Cell, kCut, kForce>(A, l, front_width(end), &A.sched->cursor[l], 0, end, s,
                          front_strided(A, l == A.level0, 0, end));
    block_tally_flush(A.stats);
}

// The kept sums of first segments in the plain schedule.
template <bool kForce>
__global__ void __launch_bounds__(256) k_add_first(const __grid_constant__ TraceArgs A)
{
    add_first(A, accumulator<kForce>(A));
}

// Resets the per-level counters of the plain schedule before the next source, whose launches
// have `warps` warps.
__global__ void k_reset_counts(Sched* sc, unsigned warps)
{
    int t = threadIdx.x;
    if (t < kNL) { sc->count[t] = 0; sc->cursor[t] = 32ull * warps; }
}

// Chooses the next phase of the persistent schedule (run by one thread, all others waiting).
__device__ __forceinline__ void next_phase(const TraceArgs& A)
{
    Sched* sc = A.sched;
    const int started = __ldcg(&sc->started);
    int l = -1;
    unsigned long long have = 0;
    // the counts of all levels are read side by side (one after the other they took 2 us)
#pragma unroll
    for (int k = 0; k < kLevels; ++k) {
        const unsigned long long c = __ldcg(&sc->count[k]);
        if (c > 0) {
            l = k;
            have = c;
        }
    }
    if (!started) {
        l = A.level0;
        have = (unsigned long long)A.base_quads * A.nsrc;
    }
    sc->started = 1;
    if (l < 0) {
        sc->done = 1;
        return;
    }
    unsigned long long take = have;
    if (l < A.lmax_glob) take = min(have, A.quad[l + 1].cap / 4);
    if (take == 0) {  // a phase must consume rays, or the schedule never ends
        atomicCAS(&A.stats->error, 0, -8);  // ART_EINTERNAL
        take = have;
    }
    const bool base = l == A.level0;
    if (base && take > 16) take -= (have - take) % 16u ? 16u - (have - take) % 16u : 0u;
    const int width = front_width(take);
    sc->phase_strided = front_strided(A, base, have - take, have);
    sc->phase_level = l;
    sc->phase_width = width;
    sc->phase_end = have;
    sc->phase_begin = have - take;
    sc->cursor[l] = (have - take) * (unsigned long long)(4 / width) + 32ull * warps_in_grid();
    sc->count[l] = have - take;
}

// Persistent schedule: all sources, all levels, one cooperative launch.
template <class Cell, bool kCut, bool kForce>
__global__ void __launch_bounds__(kTraceMaxThreads, kTraceMinBlocks) k_trace_persistent(const __grid_constant__ TraceArgs A)
{
    block_tally_init();
    Sched* sc = A.sched;
    __shared__ int s_level, s_width, s_strided, s_base_done;
    __shared__ unsigned long long s_begin, s_end;
    if (threadIdx.x == 0) s_level = -1;
    for (;;) {
        if (!grid_barrier(sc, A.stats, A.wait_ns, [&] { next_phase(A); })) break;
        if (threadIdx.x == 0) {
            s_base_done = s_level == A.level0 && s_begin == 0;  // the phase before
            s_level = __ldcg(&sc->done) ? -1 : __ldcg(&sc->phase_level);
            s_width = __ldcg(&sc->phase_width);
            s_strided = __ldcg(&sc->phase_strided);
            s_begin = __ldcg(&sc->phase_begin);
            s_end = __ldcg(&sc->phase_end);
        }
        __syncthreads();
        const int l = s_level;
        if (l >= 0) run_front<Cell, kCut, kForce>(A, l, s_width, &sc->cursor[l], s_begin, s_end, 0u, s_strided != 0);
        if (s_base_done && A.first) add_first(A, accumulator<kForce>(A));
        if (l < 0) break;
    }
    block_tally_flush(A.stats);
}

// Gamma, force and energy from the accumulator (padded layout) into the caller's SoA
// outputs (nx*ny*nz layout), four cells per thread and round.
template <class D>
__global__ void __launch_bounds__(256) k_finalize(int nx, int ny, int nz,
                                                  const D* __restrict__ acc, float gscale,
                                                  float fscale, float escale,
                                                  float* __restrict__ gamma,
                                                  float* __restrict__ force,
                                                  float* __restrict__ energy,
                                                  DevState* state, DevStats* host)
{
    finish_state(state, host);
    const unsigned ncell = (unsigned)nx * (unsigned)ny * (unsigned)nz;
    const unsigned long long step = 4ull * gridDim.x * blockDim.x;
    for (unsigned long long base = 4ull * blockIdx.x * blockDim.x + threadIdx.x; base < ncell; base += step) {
        D a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long i = base + (unsigned)k * blockDim.x;
            if (i < ncell) a[k] = __ldcs(acc + pad_of((unsigned)i, nx, ny));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long i = base + (unsigned)k * blockDim.x;
            if (i >= ncell) break;
            float G;
            if constexpr (std::is_same<D, float4>::value) {
                G = a[k].x;
                force[i] = fscale * a[k].y;
                force[(size_t)ncell + i] = fscale * a[k].z;
                force[2 * (size_t)ncell + i] = fscale * a[k].w;
            } else {
                G = a[k];
            }
            gamma[i] = gscale * G;
            if (energy) energy[i] = escale * G;
        }
    }
}

}  // namespace art
