// art_device.cuh -- device-side building blocks of the GB300 adaptive ray trace.
//
// * Distances along a ray (next face per axis, current position, split radii) are 64-bit
//   fixed-point numbers with TraceArgs::fbits fraction bits, as many as the box diagonal
//   leaves room for (51 at 512^3): a face 500 cells from the source sits within 1e-12 cells
//   of its place, an advance is one 64-bit integer add and an order decision one compare.
//   Against pairs of floats this alone took a reverse sweep bound by its instructions from
//   9.82 to 8.91 ms (128^3, 16 sources) and a forward trace bound by one deposit per crossing
//   from 83.6 to 81.9 ms (256^3, 64 sources).
// * Double-float ("df") arithmetic (an unevaluated sum hi + lo of two floats, ~44 significant
//   bits) places the start of a ray: FP64 throughput on this part is a small fraction of FP32.
// * The ray-walk state and one crossing step of Sec. 2.1 (Kim et al. 2017): next face
//   crossing per axis measured from the source, segment length, attenuation
//   dL = L (1 - e^-dtau) with dtau = chi ds (Eq. e:RT2), deposit of sum dL/chi and sum dL n
//   (Eqs. e:Erad, e:Frad), retirement at tau > tau_max or on leaving the grid, split at
//   r_max(l).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace art {

constexpr int kNL = 20;                 // level slots
constexpr int kLevels = 14;             // levels 0..13 are used
constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------------------
// double-float arithmetic
// ---------------------------------------------------------------------------------------
struct df {
    float hi, lo;
};

__device__ __forceinline__ df df_two_sum(float a, float b)
{
    float s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ df df_quick(float a, float b)  // requires |a| >= |b|
{
    float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df df_add(df a, df b)
{
    df s = df_two_sum(a.hi, b.hi);
    return df_quick(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ df df_mul(df a, df b)
{
    float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return df_quick(p, e);
}

// ---------------------------------------------------------------------------------------
// fixed-point distances
// ---------------------------------------------------------------------------------------
using fix = long long;
// "Never reached": the face distance of an axis with n_a = 0 and of faces beyond the box.
// Faces inside the box lie below 2^61 (see fraction_bits), so kFar stays apart from them and
// a face step of at most kFarStep keeps every sum below 2^63.
constexpr fix kFar = 1ll << 62;
constexpr fix kFarStep = 1ll << 61;
constexpr fix kNoEnd = 0x7fffffffffffffffll;  // end radius of a ray that ends at no radius

// Face spacing 1/|n_a| of the direction tables: m 2^(8k) with m < 2^61 in the low bits and
// the smallest such k (0..3) above them. n_a is 0 or at least 2^-24, so the product with an
// offset keeps its accuracy where the spacing itself is far beyond the box.
__device__ __forceinline__ fix encode_spacing(double spacing)
{
    unsigned long long k = 0;
    while (spacing >= 0x1p61) {
        spacing *= 0x1p-8;
        ++k;
    }
    const unsigned long long m = (unsigned long long)__double2ll_rn(spacing);
    return (fix)(m < (1ull << 61) ? m | (k << 61) : (1ull << 53) | ((k + 1) << 61));
}

// The distance to the next face from the spacing code: off * spacing for an offset of `off`
// cells (fixed-point, >= 0) along the axis; kFar when that is beyond every box. step receives
// the distance between faces, at most kFarStep. 33 <= fbits <= 59.
__device__ __forceinline__ fix face_distance(fix off, fix code, int fbits, fix& step)
{
    const unsigned k8 = 8u * (unsigned)((unsigned long long)code >> 61);
    const unsigned long long a = (unsigned long long)off;
    const unsigned long long b = (unsigned long long)code & ((1ull << 61) - 1ull);
    const unsigned long long hi = __umul64hi(a, b), lo = a * b;
    const unsigned s = (unsigned)fbits - 32u;
    const unsigned l0 = (unsigned)lo, l1 = (unsigned)(lo >> 32);
    const unsigned h0 = (unsigned)hi, h1 = (unsigned)(hi >> 32);
    const unsigned w1 = __funnelshift_l(l0, l1, k8), w2 = __funnelshift_l(l1, h0, k8),
                   w3 = __funnelshift_l(h0, h1, k8);
    const unsigned t0 = __funnelshift_r(w1, w2, s), t1 = __funnelshift_r(w2, w3, s);
    step = k8 ? kFarStep : (fix)b;
    return (hi >> ((unsigned)fbits - 2u - k8)) ? kFar : (fix)(((unsigned long long)t1 << 32) | t0);
}

// ---------------------------------------------------------------------------------------
// shared data layouts
// ---------------------------------------------------------------------------------------

// Per source: position in cell units (df split over two float4, and fixed-point) + base-ray
// luminosity and the source's l_max.
struct SrcDev {
    float4 hi;  // u_x, u_y, u_z (hi parts), L / N_ray(l0)
    float4 lo;  // u_x, u_y, u_z (lo parts), l_max (int bits)
    longlong2 xy;  // u_x, u_y (fixed-point)
    longlong2 z_;  // u_z (fixed-point), the cell that the source lies in, on a face the upper one
                   // (index in the padded layout)
};

__device__ __forceinline__ int source_cell(const SrcDev& d) { return (int)__ldg(&d.z_).y; }

// Per level constants of a trace.
struct LevelInfo {
    df r0;              // start radius of level-l rays (r_max(l-1), 0 at l0), cell units
    fix r0x, rmaxx;     // the same and the split radius r_max(l), fixed-point
    const float4* dir;     // direction table of level l: 3 float4 per pixel holding n
                           // (hi, lo) and a face spacing code per axis
    unsigned long long destroy_w;  // 4^(l_max_global - l)
};

// Forward fronts: one record per quad, the four children of a split ray, {source, pixel of
// the first child, entering L of each child (bits), tau (bits)}; two-bin traces add {Ln, taun}.
struct QuadBuf {
    uint4* rec;
    float2* recn;
    unsigned long long cap;
};

// Adjoint fronts: the same records, the slot (4 quad + child) of the quad's parent ray in the
// level above (kDone once the quad is finished), and per ray its own weighted sum (pass 1,
// double-float) and the weighted sum over its descendants.
struct AdjBuf {
    uint4* rec;
    unsigned* parent;
    float2* own;
    float* sub;
    unsigned long long cap;  // quads
};
constexpr unsigned kDone = 0xffffffffu;

// Device-resident counters of one trace.
struct DevStats {
    unsigned long long crossings, destroy, rays_total;
    unsigned long long rays_per_level[kNL];
    double escaped, dropped;
    double escaped_n, dropped_n;
    int level_reached;
    int error;
};

// Scheduler state of the persistent trace and of the plain per-level launches.
struct Sched {
    unsigned long long count[kNL];   // quads held in the level's front (a stack, top = count)
    unsigned long long cursor[kNL];  // next item (one or two rays) of the current phase / launch
    unsigned long long phase_begin, phase_end;
    int phase_level, phase_width, phase_strided, phase_kind, done, started;
    // adjoint: quads of a level whose descendants are still being swept
    unsigned long long open_begin[kNL], open_end[kNL];
    unsigned bar_count, bar_gen;
};

struct DevState {
    Sched sched;
    DevStats stats;
};

// Run by the last kernel of a trace: copies the counters to pinned host memory and leaves the
// state cleared for the next trace (a copy and a clearing of their own took 2 us each).
__device__ __forceinline__ void finish_state(DevState* state, DevStats* host)
{
    static_assert(sizeof(DevStats) % 8 == 0 && sizeof(DevState) % 8 == 0, "copied in words");
    if (blockIdx.x != 0) return;
    const unsigned long long* from = reinterpret_cast<const unsigned long long*>(&state->stats);
    unsigned long long* to = reinterpret_cast<unsigned long long*>(host);
    unsigned long long* all = reinterpret_cast<unsigned long long*>(state);
    for (unsigned i = threadIdx.x; i < sizeof(DevStats) / 8; i += blockDim.x) to[i] = from[i];
    __syncthreads();
    for (unsigned i = threadIdx.x; i < sizeof(DevState) / 8; i += blockDim.x) all[i] = 0ull;
}

// Everything the trace kernels read.
struct CellF;
struct CellW;

struct TraceArgs {
    int nx, ny, nz;
    int level0, lmax_glob;
    float tau_max;
    const float* chi;        // opacity per cell times dx (per cell length), padded layout
    const float2* chi2;      // two-bin traces: {chi_i, chi_n} per cell length, padded
    const float* srcLn;      // two-bin traces: base-ray non-ionizing luminosity per source
    const float4* rec;       // adjoint: per cell {chi, chi_H, w, 0}
    float* grad;             // adjoint gradient per cell (padded scratch)
    double* dL;              // adjoint output per source
    float4* acc;             // per-cell accumulator (sum L ds phi, sum dL n), padded
    const SrcDev* src;
    const LevelInfo* levels;
    AdjBuf adj[kNL];         // adjoint fronts
    QuadBuf quad[kNL];       // forward fronts (levels beyond l0)
    float* first;            // sums of the base rays' first segments, 8 per group of 32 rays
                             // (see keep_first); null where they are added as they come
    unsigned base_quads;     // quads of level l0 per source (3 * 4^l0)
    unsigned nsrc;
    unsigned npad;           // cells of the padded layout; cell npad is the end marker
    Sched* sched;
    DevStats* stats;
    long long wait_ns;       // bound of a grid-barrier wait (<0: give up at once)
    float gscale;            // adjoint: sigma_H * dx / dV (gamma per unit G)
    const float* srcL;       // adjoint: source luminosities (gradients scale with them)
    const CellF* recf;       // adjoint with a force term: per cell {chi, chi_H, w, 0}, {v, 0}
    const CellW* recw;       // adjoint without dust and force term: per cell {chi, w}
    fix dmax;                // d_max cutoff (kernels built for a cutoff only)
    float fscale;            // adjoint: force per unit momentum (1 / dV)
    int fbits;               // fraction bits of the fixed-point distances
    float unit;              // 2^-fbits, their unit in cells
};

// ---------------------------------------------------------------------------------------
// ray walk
// ---------------------------------------------------------------------------------------
// Per-cell record gathered at every step: the opacity alone (forward), or
// {opacity, its neutral-H part, loss weight, unused} (adjoint).
__device__ __forceinline__ float chi_of(const float4& c) { return c.x; }
// A cell record of two floats marks a two-bin trace: {chi_i, chi_n}.
template <class Cell> struct TwoBin { static constexpr bool value = false; };
template <> struct TwoBin<float2> { static constexpr bool value = true; };
__device__ __forceinline__ float4 load_cell(const float4* p) { return __ldg(p); }
// Cell record of a reverse sweep whose loss has a force term: {chi, chi_H, w, 0} and the
// force weight {v_x, v_y, v_z, 0} (32 bytes, two 16-byte gathers per step).
struct CellF {
    float4 a, b;
};
__device__ __forceinline__ float chi_of(const CellF& c) { return c.a.x; }
__device__ __forceinline__ CellF load_cell(const CellF* p) { return {__ldg(&p->a), __ldg(&p->b)}; }
// Cell record of a reverse sweep without dust and without a force term: {chi, w} (8 bytes).
// Without dust the neutral-H opacity is chi itself (both are float(n_H0 sigma_H dx)).
struct __align__(8) CellW {
    float chi, w;
};
__device__ __forceinline__ float chi_of(const CellW& c) { return c.chi; }
__device__ __forceinline__ CellW load_cell(const CellW* p)
{
    const float2 v = __ldg(reinterpret_cast<const float2*>(p));
    return {v.x, v.y};
}

// Where a ray is on its way through the grid.
struct Path {
    fix t[3];     // distance from the source to the next face on each axis
    fix d[3];     // distance between consecutive faces on each axis (1/|n_a|)
    fix tc;       // distance of the current position
    int idx;      // index of the current cell in the padded layout (sentinel ring around
                  // the grid, see pad_index)
    int ss[3];    // signed index step of a crossing on each axis
};

// An opacity coefficient (cross section times cell length) in two floats; wide marks one whose
// parts do not fit (the opacity is then formed in FP64).
struct Coef {
    float hi, lo;
    double full;
    int wide;
};

// c n to float: the product in two floats, rounded once (in FP64, at 1/64 of the FP32 rate, the
// conversions alone bounded the opacity pass: 24 us for 128^3 cells).
__device__ __forceinline__ df coef_times(const Coef& c, float n)
{
    const float p = c.hi * n;
    return {p, fmaf(c.lo, n, fmaf(c.hi, n, -p))};
}

__device__ __forceinline__ bool bad_density(float v) { return !(v >= 0.f) || isinf(v); }

// Opacity per cell length of a cell with neutral density a and total density b (0 without dust):
// neutral-H part, dust part and their sum, each rounded once from the exact value.
__device__ __forceinline__ void opacities(const Coef& sH, const Coef& sd, float a, float b,
                                          float& chi, float& chiH, float& dust)
{
    if (sH.wide | sd.wide | !(a < 1e18f) | !(b < 1e18f)) {
        const double h = (double)a * sH.full, d = (double)b * sd.full;
        chi = __double2float_rn(h + d);
        chiH = __double2float_rn(h);
        dust = __double2float_rn(d);
        return;
    }
    const df h = coef_times(sH, a), d = coef_times(sd, b);
    chiH = h.hi + h.lo;
    dust = d.hi + d.lo;
    chi = df_add(h, d).hi;
}

// Cell records are stored with a ring of sentinel cells around the nx*ny*nz grid (opacity
// < 0): cell (i, j, k) sits at (i + 1) + (nx + 2) ((j + 1) + (ny + 2) (k + 1)). A ray leaves
// the grid when the cell it steps into is a sentinel, so the walk keeps no per-axis count of
// cells left, and the cell after any crossing from inside the grid is a valid address.
__host__ __device__ __forceinline__ long long pad_index(long long i, long long j, long long k,
                                                        int nx, int ny)
{
    return (i + 1) + (long long)(nx + 2) * ((j + 1) + (long long)(ny + 2) * (k + 1));
}
constexpr float kSentinel = -1.0f;
constexpr float kEnded = -2.0f;  // opacity of the end marker, the cell after the padded layout

// Coordinates of padded cell q (see pad_index; padded grids hold fewer than 2^31 cells):
// false for the sentinel ring, else the cell's index in the caller's nx*ny*nz layout.
__device__ __forceinline__ bool unpad(unsigned q, int nx, int ny, int nz, unsigned& i)
{
    const unsigned px = (unsigned)nx + 2u, py = (unsigned)ny + 2u;
    const unsigned r = q / px;
    const int X = (int)(q - r * px) - 1;
    const int Y = (int)(r % py) - 1;
    const int Z = (int)(r / py) - 1;
    i = (unsigned)X + (unsigned)nx * ((unsigned)Y + (unsigned)ny * (unsigned)Z);
    return X >= 0 && X < nx && Y >= 0 && Y < ny && Z >= 0 && Z < nz;
}

// Runs store(q, inside, load(i)) for every padded cell q, i its index in the caller's layout
// (load runs for cells of the grid only). Four cells per thread and round keep four loads in
// flight; one at a time in a grid-stride loop had taken 17 us for 128^3 cells.
template <class Load, class Store>
__device__ __forceinline__ void each_padded_cell(int nx, int ny, int nz, Load load, Store store)
{
    const unsigned npad = (unsigned)(nx + 2) * (unsigned)(ny + 2) * (unsigned)(nz + 2);
    const unsigned long long step = 4ull * gridDim.x * blockDim.x;
    for (unsigned long long base = 4ull * blockIdx.x * blockDim.x + threadIdx.x; base < npad; base += step) {
        decltype(load(0u)) v[4] = {};
        bool in[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long q = base + (unsigned)k * blockDim.x;
            unsigned i = 0;
            in[k] = q < npad && unpad((unsigned)q, nx, ny, nz, i);
            if (in[k]) v[k] = load(i);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long q = base + (unsigned)k * blockDim.x;
            if (q < npad) store((unsigned)q, in[k], v[k]);
        }
    }
}

// Padded index of cell i of the caller's nx*ny*nz layout.
__device__ __forceinline__ unsigned pad_of(unsigned i, int nx, int ny)
{
    const unsigned r = i / (unsigned)nx, x = i - r * (unsigned)nx;
    return (unsigned)pad_index(x, r % (unsigned)ny, r / (unsigned)ny, nx, ny);
}

// Sets up the path of a ray with direction n (df) and face spacing codes (both from the
// direction table) from source position u (df, and ux fixed-point) starting at radius r0.
// Returns false if the start point lies outside the grid.
__device__ __forceinline__ bool path_start(Path& W, int nx, int ny, int nz, int fbits,
                                           const df u[3], const fix ux[3], const df n[3],
                                           const fix code[3], df r0, fix r0x)
{
    const int N[3] = {nx, ny, nz};
    int c[3];
    bool inside = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        df p = (r0.hi == 0.f) ? u[a] : df_add(u[a], df_mul(r0, n[a]));
        float f = floorf(p.hi);
        int ci = (int)f;
        if (p.hi == f && (p.lo < 0.f || (p.lo == 0.f && n[a].hi < 0.f))) ci -= 1;
        c[a] = ci;
        inside = inside && ci >= 0 && ci < N[a];
        const bool up = n[a].hi > 0.f, flat = n[a].hi == 0.f;
        const int stride = a == 0 ? 1 : (a == 1 ? nx + 2 : (nx + 2) * (ny + 2));
        W.ss[a] = flat ? 0 : (up ? stride : -stride);
        const fix face = (fix)(up ? ci + 1 : ci) << fbits;
        const fix off = up ? face - ux[a] : ux[a] - face;
        const fix t = face_distance(off > 0 ? off : 0, code[a], fbits, W.d[a]);
        W.t[a] = flat ? kFar : t;
    }
    W.tc = r0x;
    W.idx = inside ? (int)pad_index(c[0], c[1], c[2], nx, ny) : 0;
    return inside;
}

__device__ __forceinline__ float ex2_ftz(float v)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float rcp_ftz(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
constexpr float kHalfLog2e = 0.72134752f;  // log2(e) / 2: e^{-x/2} = 2^{-x kHalfLog2e}

// Arithmetic on the values of one ray (float) or of two rays side by side (float2, which this
// part adds and multiplies in one instruction).
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b)
{
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);  // exact product: one rounding
}
template <class V> __device__ __forceinline__ V vset(float v);
template <> __device__ __forceinline__ float vset<float>(float v) { return v; }
template <> __device__ __forceinline__ float2 vset<float2>(float v) { return make_float2(v, v); }
__device__ __forceinline__ float vex2(float v) { return ex2_ftz(v); }
__device__ __forceinline__ float2 vex2(float2 v) { return make_float2(ex2_ftz(v.x), ex2_ftz(v.y)); }
__device__ __forceinline__ float vrcp_max1(float v) { return rcp_ftz(fmaxf(v, 1.f)); }
__device__ __forceinline__ float2 vrcp_max1(float2 v)
{
    return make_float2(rcp_ftz(fmaxf(v.x, 1.f)), rcp_ftz(fmaxf(v.y, 1.f)));
}
// a where x < 1, else b
__device__ __forceinline__ float vbelow1(float x, float a, float b) { return x < 1.f ? a : b; }
__device__ __forceinline__ float2 vbelow1(float2 x, float2 a, float2 b)
{
    return make_float2(x.x < 1.f ? a.x : b.x, x.y < 1.f ? a.y : b.y);
}
__device__ __forceinline__ float& vget(float& v, int) { return v; }
__device__ __forceinline__ float& vget(float2& v, int j) { return j ? v.y : v.x; }
__device__ __forceinline__ float vget(const float& v, int) { return v; }
__device__ __forceinline__ float vget(const float2& v, int j) { return j ? v.y : v.x; }

// phi(x) = (1 - e^-x)/x for x >= 0. Below 1 as E sinh(y)/y with y = x/2 and E = e^{-y}, the even
// series of sinh(y)/y to y^8 (truncation < 3e-11 for y < 1/2, no cancellation); above 1 as
// (1 - E^2)/x. One exponential serves both, and both are formed: lanes never diverge. Chosen by x,
// not as the larger of the two: up to x = 2 they differ by rounding (the error of E enters them with
// opposite signs), and the larger would bias a sum of many (2e-8 of the photons absorbed there).
template <class V>
__device__ __forceinline__ V phi_of(V x)
{
    const V E = vex2(vmul(x, vset<V>(-kHalfLog2e)));
    const V x2 = vmul(x, x);
    V S = vfma(x2, vset<V>(1.f / 92897280.f), vset<V>(1.f / 322560.f));
    S = vfma(S, x2, vset<V>(1.f / 1920.f));
    S = vfma(S, x2, vset<V>(1.f / 24.f));
    S = vfma(S, x2, vset<V>(1.f));
    const V large = vmul(vfma(vmul(E, vset<V>(-1.f)), E, vset<V>(1.f)), vrcp_max1(x));
    return vbelow1(x, vmul(E, S), large);
}

// phi(x) and phi'(x) of a ray of the reverse sweep, which needs both. Below 1, with y = x/2,
// E = e^{-y} and S = sinh(y)/y: phi = E S and phi' = E (S'(y) - S) / 2, S' to y^7 (S' - S stays
// near -1, so nothing cancels); above 1, phi' = (e^{-x} - phi)/x. Chosen by x as in
// phi_of.
template <bool kDerivative, class V>
__device__ __forceinline__ V phi_dphi(V x, V& dphi)
{
    const V E = vex2(vmul(x, vset<V>(-kHalfLog2e)));
    const V y = vmul(x, vset<V>(0.5f));
    const V y2 = vmul(y, y);
    V S = vfma(y2, vset<V>(1.f / 362880.f), vset<V>(1.f / 5040.f));
    S = vfma(S, y2, vset<V>(1.f / 120.f));
    S = vfma(S, y2, vset<V>(1.f / 6.f));
    S = vfma(S, y2, vset<V>(1.f));
    const V r = vrcp_max1(x);
    const V E2 = vmul(E, E);
    const V large = vmul(vsub(vset<V>(1.f), E2), r);
    const V phi = vbelow1(x, vmul(E, S), large);
    if constexpr (kDerivative) {
        V Sp = vfma(y2, vset<V>(1.f / 45360.f), vset<V>(1.f / 840.f));
        Sp = vfma(Sp, y2, vset<V>(1.f / 30.f));
        Sp = vfma(Sp, y2, vset<V>(1.f / 3.f));
        Sp = vmul(Sp, y);
        dphi = vbelow1(x, vmul(vmul(vset<V>(0.5f), E), vsub(Sp, S)), vmul(vsub(E2, large), r));
    }
    return phi;
}

// The geometric part of a step: the segment from tc to the next face or to the end radius
// rend (split or cutoff, kNoEnd if at none), and the advance of the walk to its end; at rend
// the next cell is the end marker npad. ds is the length (cell units; unit = 2^-fbits), x is
// chi ds and key the cell of the segment; ds and x are 0 and key is `none` where there is
// nothing to deposit: the ray is no longer alive, or the length is not positive. Deposits are
// counted in ncross. walk_move_load also replaces chi by the opacity at the start of the next
// cell's record, unless the ray is no longer alive.
//
// The earliest of the three faces and the end radius is decided on the high words (2^-19
// cells at 512^3): different high words order the distances exactly. Where two are equal
// (exact ties, near ties, a face at the end radius), or the segment is too short to show in
// them (earliest() says both), the exact 64-bit comparison decides, and axes that cross within
// 2^-40 of the distance of the earliest one step together (a diagonal step). Two distances
// within that tolerance can still have different high words when they straddle a boundary; the
// walk then crosses the two faces in two steps with a segment far below the 1e-5-cell near-tie
// threshold between them, a ray the oracle flags as near-tie.
//
// Written in PTX because the predicates of the choice then also predicate the advance: from
// C++ the compiler made branches of it (15 per ray and step instead of one for both rays of a
// lane, 97.0 against 65.7 ms on 256^3 / 64 sources with four rays per lane). Each form carries
// its own advance: with the exact choice joined before a common advance, by the predicates of
// both, every step paid 18 more instructions (14.3 against 12.2 ms on 256^3 / 16 sources).
//   operands: 0-2 t, 3 tc, 4 idx, 5 ncross, 6 ds, 7 key, 8 x, 9 chi, 10-12 d, 13-15 ss,
//   16 rend, 17 unit, 18 none, 19 npad, 20 alive, 21 earliest high word
#define ART_LENGTH "cvt.rn.f32.s64 fl, mv;\n\t"
#define ART_LENGTH_PARTS \
    "cvt.rn.f32.s64 fm, m;\n\t" \
    "cvt.rn.f32.s64 fc, %3;\n\t" \
    "cvt.rni.s64.f32 at, fm;\n\t" \
    "sub.s64 at, m, at;\n\t" \
    "cvt.rn.f32.s64 gm, at;\n\t" \
    "cvt.rni.s64.f32 at, fc;\n\t" \
    "sub.s64 at, %3, at;\n\t" \
    "cvt.rn.f32.s64 gc, at;\n\t" \
    "sub.rn.f32 fm, fm, fc;\n\t" \
    "sub.rn.f32 gm, gm, gc;\n\t" \
    "add.rn.f32 fl, fm, gm;\n\t"
#define ART_MOVE_REGS \
    "{\n\t" \
    ".reg .pred p0, p1, p2, ps, po, pa;\n\t" \
    ".reg .b32 l0, l1, l2, lr, h0, h1, h2, hr, lm;\n\t" \
    ".reg .f32 fl, fm, fc, gm, gc;\n\t" \
    ".reg .b64 m, tol, d, mv, at;\n\t" \
    "setp.ne.s32 po, %20, 0;\n\t"
#define ART_MOVE_ADVANCE(LENGTH) \
    "sub.s64 mv, m, %3;\n\t" \
    LENGTH \
    "mov.b64 %3, m;\n\t" \
    "mov.f32 %6, 0f00000000;\n\t" \
    "mov.f32 %8, 0f00000000;\n\t" \
    "@pa mul.f32 %6, fl, %17;\n\t" \
    "@pa mul.f32 %8, %9, %6;\n\t" \
    "selp.b32 %7, %4, %18, pa;\n\t" \
    "@pa add.u32 %5, %5, 1;\n\t" \
    "@p0 add.s64 %0, %0, %10;\n\t" \
    "@p1 add.s64 %1, %1, %11;\n\t" \
    "@p2 add.s64 %2, %2, %12;\n\t" \
    "@p0 add.s32 %4, %4, %13;\n\t" \
    "@p1 add.s32 %4, %4, %14;\n\t" \
    "@p2 add.s32 %4, %4, %15;\n\t" \
    "@ps mov.b32 %4, %19;\n\t"
#define ART_MOVE_FAST(LENGTH) \
    ART_MOVE_REGS \
    "mov.b64 {l0, h0}, %0;\n\t" \
    "mov.b64 {l1, h1}, %1;\n\t" \
    "mov.b64 {l2, h2}, %2;\n\t" \
    "mov.b64 {lr, hr}, %16;\n\t" \
    "setp.eq.s32 p0, h0, %21;\n\t" \
    "setp.eq.s32 p1, h1, %21;\n\t" \
    "setp.eq.s32 p2, h2, %21;\n\t" \
    "setp.eq.s32 ps, hr, %21;\n\t" \
    "selp.b32 lm, l2, lr, p2;\n\t" \
    "selp.b32 lm, l1, lm, p1;\n\t" \
    "selp.b32 lm, l0, lm, p0;\n\t" \
    "mov.b64 m, {lm, %21};\n\t" \
    "mov.pred pa, po;\n\t" \
    ART_MOVE_ADVANCE(LENGTH)
#define ART_MOVE_EXACT(LENGTH) \
    ART_MOVE_REGS \
    "min.s64 m, %0, %1;\n\t" \
    "min.s64 m, m, %2;\n\t" \
    "shr.s64 tol, m, 40;\n\t" \
    "sub.s64 d, %0, m;\n\t" \
    "setp.le.s64 p0, d, tol;\n\t" \
    "sub.s64 d, %1, m;\n\t" \
    "setp.le.s64 p1, d, tol;\n\t" \
    "sub.s64 d, %2, m;\n\t" \
    "setp.le.s64 p2, d, tol;\n\t" \
    "setp.le.s64 ps, %16, m;\n\t" \
    "selp.b64 m, %16, m, ps;\n\t" \
    "setp.gt.and.s64 pa, m, %3, po;\n\t" \
    ART_MOVE_ADVANCE(LENGTH)
#define ART_MOVE_OPERANDS                                                                      \
        : "+l"(W.t[0]), "+l"(W.t[1]), "+l"(W.t[2]), "+l"(W.tc), "+r"(W.idx), "+r"(ncross),     \
          "=&f"(ds), "=&r"(key), "=&f"(x), "+f"(chi)                                           \
        : "l"(W.d[0]), "l"(W.d[1]), "l"(W.d[2]), "r"(W.ss[0]), "r"(W.ss[1]), "r"(W.ss[2]),     \
          "l"(rend), "f"(unit), "r"(none), "r"(npad), "r"((int)alive), "r"(high)

// High word of the earliest of the three faces and the end radius; exact says that the high
// words do not decide the step of a ray that is alive.
__device__ __forceinline__ int earliest(const Path& W, fix rend, bool alive, bool& exact)
{
    const int h0 = (int)(W.t[0] >> 32), h1 = (int)(W.t[1] >> 32), h2 = (int)(W.t[2] >> 32);
    const int hr = (int)(rend >> 32), hc = (int)(W.tc >> 32);
    const int a = min(h0, h1), b = max(h0, h1), c = min(h2, hr), d = max(h2, hr);
    const int first = min(a, c), second = min(max(a, c), min(b, d));
    exact = alive & ((second == first) | (first <= hc));
    return first;
}

// kExact: with the 64-bit comparison. kParts: the length is the difference of the ends' leading
// 24 bits plus that of the rest; both forms round alike but for segments that more than double
// the distance from the source, the first few of a ray.
template <bool kExact, bool kParts>
__device__ __forceinline__ void walk_move(Path& W, fix rend, float unit, float chi, bool alive,
                                          int high, int none, int npad, float& ds, float& x,
                                          int& key, unsigned& ncross)
{
    if constexpr (kExact && kParts) asm(ART_MOVE_EXACT(ART_LENGTH_PARTS) "}" ART_MOVE_OPERANDS);
    else if constexpr (kExact) asm(ART_MOVE_EXACT(ART_LENGTH) "}" ART_MOVE_OPERANDS);
    else if constexpr (kParts) asm(ART_MOVE_FAST(ART_LENGTH_PARTS) "}" ART_MOVE_OPERANDS);
    else asm(ART_MOVE_FAST(ART_LENGTH) "}" ART_MOVE_OPERANDS);
}

#define ART_MOVE_LOAD                   \
    "mad.wide.s32 at, %4, %22, %23;\n\t" \
    "@po ld.global.nc.f32 %9, [at];\n\t" \
    "}"
template <bool kExact, class Cell>
__device__ __forceinline__ void walk_move_load(Path& W, fix rend, float unit, float& chi,
                                               bool alive, int high, int none, int npad,
                                               const Cell* cells, float& ds, float& x, int& key,
                                               unsigned& ncross)
{
    if constexpr (kExact)
        asm(ART_MOVE_EXACT(ART_LENGTH) ART_MOVE_LOAD ART_MOVE_OPERANDS, "n"((int)sizeof(Cell)), "l"(cells));
    else
        asm(ART_MOVE_FAST(ART_LENGTH) ART_MOVE_LOAD ART_MOVE_OPERANDS, "n"((int)sizeof(Cell)), "l"(cells));
}

// Deposits (float or float4) across the lanes of a warp, and their sums.
__device__ __forceinline__ float shifted(float v, int off) { return __shfl_down_sync(kFull, v, off); }
__device__ __forceinline__ float4 shifted(float4 v, int off)
{
    return make_float4(shifted(v.x, off), shifted(v.y, off), shifted(v.z, off), shifted(v.w, off));
}
__device__ __forceinline__ float from_lane(float v, int lane) { return __shfl_sync(kFull, v, lane); }
__device__ __forceinline__ float4 from_lane(float4 v, int lane)
{
    return make_float4(from_lane(v.x, lane), from_lane(v.y, lane), from_lane(v.z, lane),
                       from_lane(v.w, lane));
}
__device__ __forceinline__ float across(float v, int mask) { return __shfl_xor_sync(kFull, v, mask); }
__device__ __forceinline__ float4 across(float4 v, int mask)
{
    return make_float4(across(v.x, mask), across(v.y, mask), across(v.z, mask), across(v.w, mask));
}
__device__ __forceinline__ bool is_zero(float v) { return v == 0.f; }
__device__ __forceinline__ bool is_zero(float4 v)
{
    return v.x == 0.f && v.y == 0.f && v.z == 0.f && v.w == 0.f;
}
__device__ __forceinline__ void add_to(float& a, float b) { a += b; }
__device__ __forceinline__ void add_to(float4& a, float4 b)
{
    a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
}

// sum + rest += b, the rounding error of sum collected in rest
__device__ __forceinline__ void add_pair(float& sum, float& rest, float b)
{
    const df r = df_two_sum(sum, b);
    sum = r.hi;
    rest += r.lo;
}
__device__ __forceinline__ void add_pair(float4& sum, float4& rest, float4 b)
{
    add_pair(sum.x, rest.x, b.x);
    add_pair(sum.y, rest.y, b.y);
    add_pair(sum.z, rest.z, b.z);
    add_pair(sum.w, rest.w, b.w);
}

// sum + rest; a sum that has overflowed (its error is no number then) stays as it is
__device__ __forceinline__ float with_rest(float sum, float rest)
{
    return fabsf(rest) <= 3.4e38f ? sum + rest : sum;
}
__device__ __forceinline__ float4 with_rest(float4 sum, float4 rest)
{
    return make_float4(with_rest(sum.x, rest.x), with_rest(sum.y, rest.y), with_rest(sum.z, rest.z),
                       with_rest(sum.w, rest.w));
}

// Merges the deposits of lanes that hit the same cell (runs of equal cell index in lane
// order) into the first lane of each run and takes them from the others. Used only for the first
// segments of base-level rays that are not kept for a fixed order of addition, and for their
// gradients: at l0 = 8 that is 786,432 deposits into one cell per source, whose FP32 sum the merge
// keeps accurate. Warp-uniform.
template <class D>
__device__ __forceinline__ void merge_lanes(int& cell, D& v)
{
    const unsigned lane = threadIdx.x & 31u;
    const int prev = __shfl_up_sync(kFull, cell, 1);
    const bool dup = lane > 0 && cell >= 0 && prev == cell;
    const unsigned dups = __ballot_sync(kFull, dup);
    const unsigned after = lane == 31 ? 0u : ~dups & ~((2u << lane) - 1u);
    const int run_end = after ? __ffs(after) - 1 : 32;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const D o = shifted(v, off);
        if ((int)lane + off < run_end) add_to(v, o);
    }
    if (dup) cell = -1;
}

// Adds the deposit of ray b to that of ray a where both lie in the same cell (key: the cell,
// or a negative number of the ray's own without a deposit), leaving ray b without one.
__device__ __forceinline__ void merge_pair(int key_a, float4& a, int& key_b, const float4& b,
                                           int none)
{
    asm("{\n\t.reg .pred q;\n\tsetp.eq.s32 q, %5, %4;\n\t@q add.f32 %0, %0, %6;\n\t"
        "@q add.f32 %1, %1, %7;\n\t@q add.f32 %2, %2, %8;\n\t@q add.f32 %3, %3, %9;\n\t"
        "@q mov.b32 %4, %10;\n\t}"
        : "+f"(a.x), "+f"(a.y), "+f"(a.z), "+f"(a.w), "+r"(key_b)
        : "r"(key_a), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w), "r"(none));
}

__device__ __forceinline__ void merge_pair(int key_a, float& a, int& key_b, const float& b, int none)
{
    asm("{\n\t.reg .pred q;\n\tsetp.eq.s32 q, %2, %1;\n\t@q add.f32 %0, %0, %3;\n\t"
        "@q mov.b32 %1, %4;\n\t}"
        : "+f"(a), "+r"(key_b) : "r"(key_a), "f"(b), "r"(none));
}

// One reduction into the accumulator of cell `key`, none if it is negative.
__device__ __forceinline__ void red_if(float* base, int key, float v)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ge.s32 q, %1, 0;\n\t"
                 "@q red.global.add.f32 [%0], %2;\n\t}"
                 :: "l"(base + key), "r"(key), "f"(v) : "memory");
}
__device__ __forceinline__ void red_if(float4* __restrict__ acc, int key, float4 v)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ge.s32 q, %1, 0;\n\t"
                 "@q red.global.add.v4.f32 [%0], {%2, %3, %4, %5};\n\t}"
                 :: "l"(acc + key), "r"(key), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// ---------------------------------------------------------------------------------------
// helpers shared by the forward and backward kernels
// ---------------------------------------------------------------------------------------
// Threads per block of the trace kernels at most: one block of 20 warps per SM (65536 / 640 =
// 102 registers a thread, 96 in steps of eight: two walks), so that a grid barrier has 152 arrivals and not 760. 24
// warps (80 registers) gain 5 % at 256^3 and lose 2 % at 512^3 and 3 % in the sweep.
constexpr int kTraceMaxThreads = 640;
constexpr int kTraceMinBlocks = 1;
// Steps between checks whether a warp still has rays.
constexpr int kCheckSteps = 4;

// Tallies of a block: photon sums per thread (no atomics while rays end), counters per warp
// or per level. Reduced once, when the kernel ends.
struct BlockTally {
    double escaped[kTraceMaxThreads], dropped[kTraceMaxThreads];
    double escaped_n[kTraceMaxThreads], dropped_n[kTraceMaxThreads];
    unsigned long long crossings, destroy;
    unsigned long long rays[kNL];
};

__device__ __forceinline__ BlockTally& block_tally()
{
    __shared__ BlockTally t;
    return t;
}

__device__ __forceinline__ void block_tally_init()
{
    BlockTally& T = block_tally();
    const int i = threadIdx.x;
    T.escaped[i] = T.dropped[i] = T.escaped_n[i] = T.dropped_n[i] = 0.0;
    if (i < kNL) T.rays[i] = 0ull;
    if (i == 0) T.crossings = T.destroy = 0ull;
    __syncthreads();
}

__device__ __forceinline__ void block_tally_flush(DevStats* st)
{
    BlockTally& T = block_tally();
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = threadIdx.x; i < (int)blockDim.x; i += 32) {
        v[0] += T.escaped[i];
        v[1] += T.dropped[i];
        v[2] += T.escaped_n[i];
        v[3] += T.dropped_n[i];
    }
    double* out[4] = {&st->escaped, &st->dropped, &st->escaped_n, &st->dropped_n};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_down_sync(kFull, v[k], off);
        if (threadIdx.x == 0 && v[k] != 0.0) atomicAdd(out[k], v[k]);
    }
    if (threadIdx.x == 0) {
        if (T.crossings) atomicAdd(&st->crossings, T.crossings);
        if (T.destroy) atomicAdd(&st->destroy, T.destroy);
    }
    if (threadIdx.x < kNL && T.rays[threadIdx.x]) {
        atomicAdd(&st->rays_per_level[threadIdx.x], T.rays[threadIdx.x]);
        atomicAdd(&st->rays_total, T.rays[threadIdx.x]);
        atomicMax(&st->level_reached, (int)threadIdx.x);
    }
}

// Sum of a few floats in two floats, for the tallies.
__device__ __forceinline__ void df_accumulate(df& s, float v)
{
    const df r = df_two_sum(s.hi, v);
    s.hi = r.hi;
    s.lo += r.lo;
}

// Items of a front are taken 32 at a time, the first by the warp's place in the grid (the warps of
// an SM far apart, so that a small front spreads over the chip), further ones from a cursor
// that starts behind those: a front of one round costs no atomics, where one per warp on one
// address had taken microseconds.
__device__ __forceinline__ unsigned warps_in_grid() { return gridDim.x * (blockDim.x >> 5); }

// Place of this warp in the grid: the warps of an SM are far apart.
__device__ __forceinline__ unsigned warp_in_grid() { return (threadIdx.x >> 5) * gridDim.x + blockIdx.x; }

struct Batches {
    unsigned long long* cursor;
    unsigned next, items;
    bool first;
    __device__ __forceinline__ Batches(unsigned long long* c, unsigned begin, unsigned n)
        : cursor(c), next(begin + 32u * warp_in_grid()), items(n),
          first(true) {}
    // First item of the warp's next batch, or a value >= items when there is none. Warp-uniform.
    __device__ __forceinline__ unsigned take(unsigned begin)
    {
        if (first) {
            first = false;
            return next;
        }
        if (begin + 32u * warps_in_grid() >= items) return items;
        unsigned b = 0;
        if ((threadIdx.x & 31u) == 0)
            b = (unsigned)min(atomicAdd(cursor, 32ull), (unsigned long long)items);
        return __shfl_sync(kFull, b, 0);
    }
};

// Rays per lane for a front of `quads` quads: one while that fits the chip's warps in one
// round (latency counts there, and a step of one ray is shorter), else two. The optimum is flat:
// with the line at two or four times as many rays 128^3 / 1 source takes 276 instead of 269 us and
// an odd box of two bins 408 instead of 398 us; at half as many 273 and 402 us.
__device__ __forceinline__ int front_width(unsigned long long quads)
{
    return 4 * quads <= (unsigned long long)gridDim.x * blockDim.x ? 1 : 2;
}

// Where a ray of a level with split radius rmax ends: at rmax if it can split and (kCut) at
// the d_max cutoff, whichever comes first; at equal radii the cut wins.
template <bool kCut>
__device__ __forceinline__ fix end_radius(bool splits, fix rmax, fix dmax)
{
    const fix r = splits ? rmax : kNoEnd;
    return kCut ? min(r, dmax) : r;
}
// Whether a ray that reached its end radius splits there (else the cutoff ended it).
template <bool kCut>
__device__ __forceinline__ bool splits_at_end(bool splits, fix rmax, fix dmax)
{
    return !kCut || (splits && rmax < dmax);
}

// One entry of a direction table: n (df) and the face spacing code per axis.
__device__ __forceinline__ void load_direction(const float4* e, df n[3], fix code[3])
{
    const float4 e0 = __ldg(e), e1 = __ldg(e + 1);
    const longlong2 e2 = __ldg(reinterpret_cast<const longlong2*>(e + 2));
    n[0] = {e0.x, e0.w};
    n[1] = {e0.y, e1.x};
    n[2] = {e0.z, e1.y};
    code[0] = (fix)(((unsigned long long)__float_as_uint(e1.w) << 32) | __float_as_uint(e1.z));
    code[1] = e2.x;
    code[2] = e2.y;
}

// Grid-wide barrier for a cooperative launch. Every wait is bounded by wait_ns of
// %globaltimer; on expiry the block records ART_ETIMEOUT and the barrier returns false.
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The block that arrives last runs `last` (one thread) before it releases the others.
template <class F>
__device__ __forceinline__ bool grid_barrier(Sched* sc, DevStats* st, long long wait_ns, F last)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        unsigned g, arrived;
        asm volatile("ld.relaxed.gpu.u32 %0, [%1];" : "=r"(g) : "l"(&sc->bar_gen) : "memory");
        // release this block's writes, acquire those of the blocks before it
        asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], 1;"
                     : "=r"(arrived) : "l"(&sc->bar_count) : "memory");
        if (arrived + 1u == gridDim.x) {
            last();
            sc->bar_count = 0u;
            asm volatile("st.release.gpu.u32 [%0], %1;" :: "l"(&sc->bar_gen), "r"(g + 1u) : "memory");
        } else {
            const unsigned long long t0 = global_ns();
            for (;;) {
                unsigned now;
                asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(now) : "l"(&sc->bar_gen) : "memory");
                if (now != g) break;
                if (wait_ns < 0 || (long long)(global_ns() - t0) > wait_ns) {
                    atomicCAS(&st->error, 0, -4);  // ART_ETIMEOUT
                    ok = 0;
                    break;
                }
            }
        }
        if (*((volatile int*)&st->error) != 0) ok = 0;
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

}  // namespace art
