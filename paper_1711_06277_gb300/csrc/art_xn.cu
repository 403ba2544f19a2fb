// art_xn.cu -- neutral-fraction update (Sec. 2.3, Eqs. e:xn2 and e:xn3) and the substep
// size of Eq. e:dtss, elementwise over cells.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <mutex>

#include "art.h"
#include "art_device.cuh"

namespace {

using art::df;
using art::df_add;
using art::df_mul;
using art::df_quick;
using art::df_two_sum;

// Eq. e:xn3: the electron density is held at n_H (1 - x0) over dt, which makes Eq. e:xn
// linear; the solution relaxes to x_eq0 = a/(Gamma + a), a = alpha n_e, on t = 1/(Gamma + a).
__device__ __forceinline__ float xn_b(float x0, float gam, float nH, float alpha, float dt)
{
    const float a = alpha * nH * (1.f - x0);
    const float rate = gam + a;
    if (!(rate > 0.f)) return x0;
    const float xeq = a / rate;
    return xeq + (x0 - xeq) * __expf(-dt * rate);
}

// Eq. e:xn2: exact solution of the quadratic rate equation; for Gamma = 0 the closed form
// of the shielded cell. FP64, for cells outside the range of xn_a.
__device__ __noinline__ float xn_a_wide(float x0, float gam, float nH, float alpha, float dt)
{
    const double a = (double)alpha * nH;
    if (!(gam > 0.f)) {
        const double q = (1.0 - x0) * a * dt;
        return (float)((x0 + q) / (1.0 + q));
    }
    const double g = gam;
    const double xeq = 2.0 * a / (g + 2.0 * a + sqrt(g * g + 4.0 * a * g));
    const double xp = 1.0 / xeq;
    const double K = exp(-(xp - xeq) * dt * a);
    return (float)(xeq + (xp - xeq) * (x0 - xeq) * K / ((xp - x0) + (x0 - xeq) * K));
}

__device__ __forceinline__ df df_scale(df a, float pow2) { return {a.hi * pow2, a.lo * pow2}; }
__device__ __forceinline__ df df_sel(bool c, df a, df b) { return {c ? a.hi : b.hi, c ? a.lo : b.lo}; }

// a / b to about 2^-44: one correction of the quotient of the leading parts
__device__ __forceinline__ df df_div(df a, df b)
{
    const float y = art::rcp_ftz(b.hi);
    const float q = a.hi * y;
    const float p = q * b.hi;
    const float e = fmaf(q, b.hi, -p);
    const float r = fmaf(-q, b.lo, ((a.hi - p) - e) + a.lo);
    return df_quick(q, r * y);
}

__device__ __forceinline__ df df_sqrt(df a)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a.hi));
    const float s = a.hi * y;
    const float r = fmaf(-s, s, a.hi) + a.lo;
    return df_quick(s, 0.5f * r * y);
}

// e^-z = 2^-n (1 + u) for 0 <= z <= 80: z = n ln 2 + f, |f| <= ln(2)/2 with ln 2 in three parts
// (Cody & Waite 1980: the first, floor(2^12 ln 2) 2^-12, short enough for exact products), and
// u = e^-f - 1 by its series, the leading five terms in two floats, the rest (below 5e-5 of u)
// in one.
__device__ __forceinline__ void exp_neg(df z, float& pow2, df& u)
{
    const float n = rintf(z.hi * 1.44269504f);
    df f = df_two_sum(fmaf(-n, 0.693115234375f, z.hi), z.lo);
    f = df_add(f, df_mul({-n, 0.f}, {3.194618329871446e-05f, 1.6465949697480609e-12f}));
    const df g = {-f.hi, -f.lo};
    float t = fmaf(g.hi, 1.f / 3628800.f, 1.f / 362880.f);
    t = fmaf(t, g.hi, 1.f / 40320.f);
    t = fmaf(t, g.hi, 1.f / 5040.f);
    t = fmaf(t, g.hi, 1.f / 720.f);
    t = fmaf(t, g.hi, 1.f / 120.f);
    df s = df_add({1.f / 24.f, (float)(1.0 / 24.0 - (double)(1.f / 24.f))}, {t * g.hi, 0.f});
    s = df_add({1.f / 6.f, (float)(1.0 / 6.0 - (double)(1.f / 6.f))}, df_mul(s, g));
    s = df_add({0.5f, 0.f}, df_mul(s, g));
    s = df_add({1.f, 0.f}, df_mul(s, g));
    u = df_mul(s, g);
    pow2 = __int_as_float((127 - (int)n) << 23);
}

// Eq. e:xn2 in pairs of floats (relative error about 2^-38, so that the rounding of the result
// to one float is all that shows: the error against 64 bits is that of the FP64 form, 3.6e-8
// of the 2-norm). Bound by FP32 issue; in FP64, at 1/64 of the FP32 rate, the update of 2^24
// cells took 2.82 ms, now 0.21 ms. With
//   r = (g^2 + 4 a g)^(1/2), h = g + 2a + r, x_eq = 2a/h, 1 - x_eq = (g + r)/h,
//   K = e^{-r dt}, B = x0 - x_eq
// (the second root is x_p = 1/x_eq = h/2a and x_p - x_eq = r/a) the solution is
//   x_eq + r B K / ((g + r)/2 + a (1 - x0) + a B K)              for B > 0,
//   (x0 r + (h/2) (-B) (1 - K)) / (r + a (-B) (1 - K))           for B <= 0,
// sums of positive terms both. a and g are scaled by a power of two, which leaves the
// solution unchanged with dt scaled back.
__device__ __forceinline__ float xn_a(float x0, float gam, float nH, float alpha, float dt)
{
    df a;
    a.hi = alpha * nH;
    a.lo = fmaf(alpha, nH, -a.hi);
    const df y0 = df_two_sum(1.f, -x0);
    const bool in = a.hi > 1e-25f && a.hi < 1e25f && dt > 1e-25f && dt < 1e25f && x0 >= 0.f && x0 <= 1.f;
    if (!(gam > 0.f)) {
        const df ad = df_mul(a, {dt, 0.f});
        if (!(in && ad.hi > 1e-25f && ad.hi < 1e25f)) return xn_a_wide(x0, gam, nH, alpha, dt);
        const df q = df_mul(y0, ad);
        return df_div(df_add({x0, 0.f}, q), df_add({1.f, 0.f}, q)).hi;
    }
    const float m = fmaxf(a.hi, gam);
    const int e = (__float_as_int(m) >> 23) - 127;
    // (the exponents are bounded before the scale is formed)
    const float scale = __int_as_float((127 - max(min(e, 100), -100)) << 23);
    const float back = __int_as_float((127 + max(min(e, 100), -100)) << 23);
    a = df_scale(a, scale);
    const float g = gam * scale, d = dt * back;
    if (!(in && abs(e) < 100 && a.hi > 1e-12f && g > 1e-12f && d > 1e-18f && d < 1e18f))
        return xn_a_wide(x0, gam, nH, alpha, dt);
    const df g1 = {g, 0.f};
    const df r = df_sqrt(df_mul(df_add(g1, df_scale(a, 4.f)), g1));
    const df gr = df_add(g1, r);
    const df a2 = df_scale(a, 2.f);
    const df h = df_add(gr, a2);
    const df xeq = df_div(a2, h);
    // B from the side on which its terms are small
    const bool high = x0 > 0.5f;
    const df om = df_div(gr, h);
    df B = df_add(df_sel(high, om, {x0, 0.f}), df_sel(high, {-y0.hi, -y0.lo}, {-xeq.hi, -xeq.lo}));
    const bool pos = B.hi > 0.f;
    if (!pos) B = {-B.hi, -B.lo};
    const df z = df_mul(r, {d, 0.f});
    const bool gone = z.hi > 80.f;  // K below 2e-35 of the other terms
    float pow2;
    df u;
    exp_neg(df_sel(gone, {80.f, 0.f}, z), pow2, u);
    // K = 2^-n + 2^-n u, or 1 - K
    if (!pos) pow2 = -pow2;
    df k = df_add(df_two_sum(pos ? 0.f : 1.f, pow2), df_scale(u, pow2));
    if (gone) k = {pos ? 0.f : 1.f, 0.f};
    const df W = df_mul(B, k);
    const df rest = df_add(df_scale(gr, 0.5f), df_mul(a, y0));
    const df den = df_add(df_sel(pos, rest, r), df_mul(a, W));
    const df hw = df_mul(df_sel(pos, r, df_scale(h, 0.5f)), W);
    const df num = pos ? hw : df_add(df_mul({x0, 0.f}, r), hw);
    const df x = df_div(num, den);
    return pos ? df_add(xeq, x).hi : x.hi;
}

template <int kMethod>
__device__ __forceinline__ float xn_one(float x0, float g, float n, float alpha, float dt)
{
    const float x = kMethod == 0 ? xn_b(x0, g, n, alpha, dt) : xn_a(x0, g, n, alpha, dt);
    return fminf(fmaxf(x, 0.f), 1.f);
}

// Cells [0, ncell), four at a time where all arrays are aligned to 16 bytes (vec) and one at a
// time for the rest. HBM bound with method b: 20 bytes per cell. One 4-byte load per array and
// thread in flight ran at 3.9 TB/s (682 us for 2^27 cells), one vector per array at 6.9 (390 us).
template <int kMethod>
__global__ void __launch_bounds__(256) k_xn_update(long long ncell, bool vec,
                                                   const float* __restrict__ gamma,
                                                   const float* __restrict__ nH,
                                                   float* __restrict__ xn, float* __restrict__ nH0,
                                                   float alpha, float dt)
{
    const long long step = (long long)gridDim.x * blockDim.x;
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long nvec = vec ? ncell / 4 : 0;
    for (long long i = first; i < nvec; i += step) {
        const float4 n = __ldcs(reinterpret_cast<const float4*>(nH) + i);
        const float4 x0 = __ldcs(reinterpret_cast<const float4*>(xn) + i);
        const float4 g = __ldcs(reinterpret_cast<const float4*>(gamma) + i);
        const float4 x = make_float4(xn_one<kMethod>(x0.x, g.x, n.x, alpha, dt),
                                     xn_one<kMethod>(x0.y, g.y, n.y, alpha, dt),
                                     xn_one<kMethod>(x0.z, g.z, n.z, alpha, dt),
                                     xn_one<kMethod>(x0.w, g.w, n.w, alpha, dt));
        reinterpret_cast<float4*>(xn)[i] = x;
        if (nH0)
            reinterpret_cast<float4*>(nH0)[i] =
                make_float4(x.x * n.x, x.y * n.y, x.z * n.z, x.w * n.w);
    }
    for (long long i = 4 * nvec + first; i < ncell; i += step) {
        const float n = nH[i];
        const float x = xn_one<kMethod>(xn[i], gamma[i], n, alpha, dt);
        xn[i] = x;
        if (nH0) nH0[i] = x * n;
    }
}

__device__ __forceinline__ float dt_one(float m, float n, float x, float g, float alpha)
{
    const float ne = n * (1.f - x);
    const float d = fabsf(x * n * g - alpha * ne * ne);
    return d > 0.f ? fminf(m, n / d) : m;
}

// Per-block minimum of n_H / |I - R| (I = x n_H Gamma, R = alpha (n_H (1 - x))^2), four cells at
// a time where the arrays are aligned to 16 bytes (vec).
__global__ void k_dt_partial(long long ncell, bool vec, const float* __restrict__ gamma,
                             const float* __restrict__ nH, const float* __restrict__ xn,
                             float alpha, float* __restrict__ part)
{
    __shared__ float s_min[32];
    float m = INFINITY;
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long step = (long long)gridDim.x * blockDim.x;
    const long long nvec = vec ? ncell / 4 : 0;
    for (long long i = first; i < nvec; i += step) {
        const float4 n = reinterpret_cast<const float4*>(nH)[i];
        const float4 x = reinterpret_cast<const float4*>(xn)[i];
        const float4 g = reinterpret_cast<const float4*>(gamma)[i];
        m = dt_one(m, n.x, x.x, g.x, alpha);
        m = dt_one(m, n.y, x.y, g.y, alpha);
        m = dt_one(m, n.z, x.z, g.z, alpha);
        m = dt_one(m, n.w, x.w, g.w, alpha);
    }
    for (long long i = 4 * nvec + first; i < ncell; i += step)
        m = dt_one(m, nH[i], xn[i], gamma[i], alpha);
    for (int off = 16; off > 0; off >>= 1) m = fminf(m, __shfl_down_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) s_min[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = threadIdx.x < (blockDim.x + 31) / 32 ? s_min[threadIdx.x] : INFINITY;
        for (int off = 16; off > 0; off >>= 1) m = fminf(m, __shfl_down_sync(0xffffffffu, m, off));
        if (threadIdx.x == 0) part[blockIdx.x] = m;
    }
}

__global__ void k_dt_final(int nparts, const float* __restrict__ part, double C, double* out)
{
    __shared__ float s_min[32];
    float m = INFINITY;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) m = fminf(m, part[i]);
    for (int off = 16; off > 0; off >>= 1) m = fminf(m, __shfl_down_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) s_min[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = threadIdx.x < (blockDim.x + 31) / 32 ? s_min[threadIdx.x] : INFINITY;
        for (int off = 16; off > 0; off >>= 1) m = fminf(m, __shfl_down_sync(0xffffffffu, m, off));
        if (threadIdx.x == 0) *out = isinf(m) ? (double)INFINITY : C * (double)m;
    }
}

constexpr int kDtBlocks = 1024;

}  // namespace

// ---------------------------------------------------------------------------------------
// Allocation-free variant of art_dt_substep (no counterpart in the paper).
//
// Some callers cannot call cudaMalloc: code embedded in a host framework that owns all of
// the device memory through its own pool, where a fresh allocation fails or fragments that
// pool, and latency-critical loops that cannot afford the implicit device synchronization of
// cudaMalloc/cudaFree. For them the per-block partial minima live in this fixed array,
// which every GPU that loads the library keeps for the life of the process: one float per
// 256-cell tile, so inputs of up to ART_DT_STATIC_MAX_CELLS cells.
// ---------------------------------------------------------------------------------------
namespace {

constexpr int kStaticTiles = 65536;  // ART_DT_STATIC_MAX_CELLS / 256
static __device__ __align__(256) float g_dt_partials[kStaticTiles];

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
float* g_static_ptr[kMaxDevices] = {};

// Device address of g_dt_partials on the current device, looked up once per device. In
// host code the symbol's name is only a host-side stand-in and must never reach a kernel.
int static_partials(float** out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ART_ECUDA;
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_dt_partials) != cudaSuccess || !p) return ART_ECUDA;
        g_static_ptr[dev] = static_cast<float*>(p);
    }
    *out = g_static_ptr[dev];
    return ART_OK;
}

}  // namespace

extern "C" {

int art_xn_update(void* stream, long long ncell, const float* d_gamma, const float* d_nH,
                  float* d_xn, float* d_nH0, double alpha_B, double dt, int method)
{
    if (ncell < 0 || (ncell > 0 && (!d_gamma || !d_nH || !d_xn))) return ART_EINVAL;
    if (!(alpha_B > 0.0) || !(dt >= 0.0) || !std::isfinite(dt) || (method != 0 && method != 1))
        return ART_EINVAL;
    if (ncell == 0) return ART_OK;
    const size_t bits = (size_t)d_gamma | (size_t)d_nH | (size_t)d_xn | (size_t)d_nH0;
    const bool vec = bits % 16 == 0;
    // one vector per thread: 2^24 cells and more need no loop (the grid is capped far above)
    const long long work = vec ? (ncell + 3) / 4 : ncell;
    const int blocks = (int)std::min<long long>((work + 255) / 256, 1ll << 24);
    auto kern = method == 0 ? k_xn_update<0> : k_xn_update<1>;
    kern<<<blocks, 256, 0, (cudaStream_t)stream>>>(ncell, vec, d_gamma, d_nH, d_xn, d_nH0,
                                                   (float)alpha_B, (float)dt);
    return cudaGetLastError() == cudaSuccess ? ART_OK : ART_ECUDA;
}

long long art_dt_scratch_bytes(long long ncell)
{
    (void)ncell;
    return (long long)kDtBlocks * (long long)sizeof(float);
}

int art_dt_substep(void* stream, long long ncell, const float* d_gamma, const float* d_nH,
                   const float* d_xn, double alpha_B, double C, void* d_scratch, double* d_dt)
{
    if (ncell <= 0 || !d_gamma || !d_nH || !d_xn || !d_scratch || !d_dt) return ART_EINVAL;
    if (!(alpha_B > 0.0) || !(C > 0.0)) return ART_EINVAL;
    long long want = (ncell + 255) / 256;
    const int blocks = (int)(want < kDtBlocks ? want : kDtBlocks);
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bits = (size_t)d_gamma | (size_t)d_nH | (size_t)d_xn;
    k_dt_partial<<<blocks, 256, 0, s>>>(ncell, bits % 16 == 0, d_gamma, d_nH, d_xn, (float)alpha_B,
                                        (float*)d_scratch);
    k_dt_final<<<1, 1024, 0, s>>>(blocks, (const float*)d_scratch, C, d_dt);
    return cudaGetLastError() == cudaSuccess ? ART_OK : ART_ECUDA;
}

int art_dt_substep_static(void* stream, long long ncell, const float* d_gamma, const float* d_nH,
                          const float* d_xn, double alpha_B, double C, double* d_dt)
{
    if (ncell <= 0 || !d_gamma || !d_nH || !d_xn || !d_dt) return ART_EINVAL;
    if (ncell > ART_DT_STATIC_MAX_CELLS) return ART_EINVAL;  // beyond the fixed scratch
    if (!(alpha_B > 0.0) || !(C > 0.0)) return ART_EINVAL;
    float* partials = nullptr;
    const int rc = static_partials(&partials);
    if (rc != ART_OK) return rc;
    // one tile of 256 cells per block: every partial read below is written first by its
    // block in this call, so nothing carries over from an earlier call
    const int tiles = (int)((ncell + 255) / 256);
    cudaStream_t s = (cudaStream_t)stream;
    // (a cell per thread: four at a time, a tile would use a quarter of its block's threads)
    k_dt_partial<<<tiles, 256, 0, s>>>(ncell, false, d_gamma, d_nH, d_xn, (float)alpha_B, partials);
    k_dt_final<<<1, 1024, 0, s>>>(tiles, partials, C, d_dt);
    return cudaGetLastError() == cudaSuccess ? ART_OK : ART_ECUDA;
}

}  // extern "C"
