// Cone-beam reconstruction of simulated scans (Section 3.5 reconstructs the
// simulated projections with an FDK algorithm).  Feldkamp-Davis-Kress for the
// circular orbit of Section 2.1 with the imager opposite the source, in the
// textbook form (Kak & Slaney, equally spaced fan beam, Feldkamp's cone
// weighting):
//   * line integrals g = -ln(I / I0) against the air scan I0;
//   * virtual detector at the isocentre (a = u SAD / SDD, b = v SAD / SDD,
//     spacing tau = du SAD / SDD), cosine weight SAD / sqrt(SAD^2 + a^2 + b^2);
//   * Ram-Lak ramp along each row as a linear convolution with zeros outside
//     the row, times the 1/2 of the full-scan fan-beam formula:
//     Qf(n) = (1 / (2 tau)) (q(n) / 4 - sum_{odd d} q(n - d) / (pi d)^2);
//   * voxel-driven backprojection f(x) = sum_beta dbeta (SAD / depth)^2
//     Qf(a(x), b(x)), depth = SAD + x.n, bilinear on the pixel-centre grid,
//     zero outside the detector.
// The filter is a dense row convolution (nu^2 / 2 FMAs per row) from shared
// memory with register tiles; the backprojection gathers 4 detector samples per voxel
// and view from L1 / L2 and keeps a few voxels of a column in registers, so the
// per-view geometry (depth, u, weight) is computed once per column.
#include <algorithm>
#include <cmath>
#include <functional>

#include "fdk_filter.h"
#include "fdk_rows.h"
#include "gdrr_internal.cuh"

namespace gdrr {
namespace {

constexpr int BP_MAX_ANGLES = 128;     // views per backprojection launch (kernel parameters)
constexpr int BP_ZT = 4;               // voxels of a column per thread
constexpr int BP_BX = 32, BP_BY = 8;   // voxels of a block in x and y, by warps of 8 x 4
constexpr int BP_WX = 8;

struct FilterParams {
    int nu, nv;
    float mag_du, mag_dv;   // virtual-detector spacings tau_u, tau_v (mm)
    float sad;
    float scale;            // 1 / (2 tau_u)
};

// The convolution of one parity is a product with a Toeplitz matrix: outputs
// n = 2a + par take sources k = 2b + 1 - par (odd offsets only) with the
// coefficient T[a - b + nb], one signed table per parity.  A thread owns FO
// outputs (consecutive a) of FR rows: as b advances by one, its FO
// coefficients slide by one slot, so a step loads one coefficient and, two
// sources at a time, the FR rows' samples, for FO x FR FMAs, packed in pairs
// of rows (fma.rn.f32x2).  The rows sit in shared memory weighted, split by
// parity and interleaved in pairs, zero beyond the row; the table is padded by one slot in FO so that
// the lanes of a warp (FO slots apart) read different banks.
//
// Bound: FP32 FMA (nu^2 / 2 per row; 18.1 G for 360 views of 512 x 384: 0.49 ms
// at 128 per SM and cycle) and the rows' weighting before it: 0.88 ms.  One row
// per block and 4 outputs per thread took 2.6 ms at the full shared-memory
// rate; 8 rows per thread (2 blocks per SM) 0.95 ms, 2 rows 0.85 ms.
constexpr int FL = 16;                          // loads of a lane under way at a time

__global__ void __launch_bounds__(FILTER_BLOCK, FILTER_BLOCKS_PER_SM) fdk_filter_kernel(const FilterParams p, const FilterShape f,
                                                                    int64_t n_rows, const float* __restrict__ g,
                                                                    float* __restrict__ out) {
    extern __shared__ __align__(16) float sm[];
    const int nu = p.nu;
    float* q = sm;                                            // [2][rows][stride]
    float* tab = sm + (size_t)2 * f.rows * f.stride;          // [2][tab]
    const int64_t r0 = (int64_t)blockIdx.x * f.rows;
    const int rows = (int)min((int64_t)f.rows, n_rows - r0);
    // T[a - b + nb] of parity par: offset n - k = 2 (a - b) + 2 par - 1
    for (int i = threadIdx.x; i < 2 * (2 * f.nb + FO); i += FILTER_BLOCK) {
        const int par = i / (2 * f.nb + FO), j = i - par * (2 * f.nb + FO);
        const float pd = 3.14159265358979f * (float)(2 * (j - f.nb) + 2 * par - 1);
        tab[par * f.tab + filter_pad(j)] = -1.0f / (pd * pd);
    }
    for (int r = threadIdx.x >> 5; r < f.rows; r += FILTER_BLOCK / 32) {
        const float b = ((float)((r0 + r) % p.nv) + 0.5f - 0.5f * (float)p.nv) * p.mag_dv;
        const float sad2b2 = p.sad * p.sad + b * b;
        const float* gr = g + (r0 + r) * nu;
        for (int k0 = threadIdx.x & 31; k0 < 2 * f.nb; k0 += 32 * FL) {
            float v[FL];                                      // FL loads under way at a time
#pragma unroll
            for (int i = 0; i < FL; ++i) v[i] = (r < rows && k0 + 32 * i < nu) ? __ldcs(gr + k0 + 32 * i) : 0.0f;
#pragma unroll
            for (int i = 0; i < FL; ++i) {
                const int k = k0 + 32 * i;
                const float a = ((float)k + 0.5f - 0.5f * (float)nu) * p.mag_du;
                if (k < 2 * f.nb)
                    q[((size_t)((k & 1) * (f.rows / 2) + (r >> 1)) * f.stride + (k >> 1)) * 2 + (r & 1)] =
                        v[i] * (p.sad / sqrtf(sad2b2 + a * a));
            }
        }
    }
    __syncthreads();
    // this block's part of the rows' tasks
    const int per_part = (filter_tasks(f) + f.parts - 1) / f.parts, first = blockIdx.y * per_part;
    const int tasks = min(filter_tasks(f), first + per_part);
    for (int task = first + threadIdx.x; task < tasks; task += FILTER_BLOCK) {
        const int o = task % f.oct, par = (task / f.oct) & 1, rg = task / (2 * f.oct);
        const uint64_t* q2 = reinterpret_cast<const uint64_t*>(q);            // one sample of two rows
        const uint64_t* own = q2 + (size_t)(par * (f.rows / 2) + rg * (FR / 2)) * f.stride + o * FO;
        const uint64_t* src = q2 + (size_t)((1 - par) * (f.rows / 2) + rg * (FR / 2)) * f.stride;
        uint64_t acc[FR / 2][FO];
#pragma unroll
        for (int r = 0; r < FR / 2; ++r)
#pragma unroll
            for (int j = 0; j < FO; ++j) acc[r][j] = fma2(twice(0.25f), own[r * f.stride + j], 0ull);
        // w[(j - b) mod FO] holds T[o FO + j - b + nb], twice
        const float* t = tab + par * f.tab + filter_pad(o * FO + f.nb);
        uint64_t w[FO];
#pragma unroll
        for (int j = 0; j < FO; ++j) w[j] = twice(t[j]);
        for (int b0 = 0; b0 < f.nb; b0 += FO) {
            t -= FO + 1;                                      // the padded slot of FO coefficients further down
#pragma unroll
            for (int h = 0; h < FO; h += 2) {
                ulonglong2 s[FR / 2];
#pragma unroll
                for (int r = 0; r < FR / 2; ++r) s[r] = *reinterpret_cast<const ulonglong2*>(src + r * f.stride + b0 + h);
#pragma unroll
                for (int b = h; b < h + 2; ++b) {
#pragma unroll
                    for (int r = 0; r < FR / 2; ++r)
#pragma unroll
                        for (int j = 0; j < FO; ++j)
                            acc[r][j] = fma2(b == h ? s[r].x : s[r].y, w[(j - b + FO) % FO], acc[r][j]);
                    w[FO - 1 - b] = twice(t[FO - 1 - b]);     // enters as the next source's first coefficient
                }
            }
        }
#pragma unroll
        for (int r = 0; r < FR / 2; ++r)
#pragma unroll
            for (int j = 0; j < FO; ++j) {
                const int n = 2 * (o * FO + j) + par;
                const float2 v = unpack2(acc[r][j]);
                if (n < nu) {
                    if (rg * FR + 2 * r < rows) out[(r0 + rg * FR + 2 * r) * nu + n] = p.scale * v.x;
                    if (rg * FR + 2 * r + 1 < rows) out[(r0 + rg * FR + 2 * r + 1) * nu + n] = p.scale * v.y;
                }
            }
    }
}

struct BpParams {
    int nx, ny, nz, nu, nv;
    float x0, y0, z0;        // first voxel centre (mm)
    float dx, dy, dz;
    float sad;
    float inv_tau_u, inv_tau_v;
    float hu, hv;            // nu / 2 - 1/2, nv / 2 - 1/2
    float d_beta;
    int n_ang;
    int accumulate;          // 1: add to the volume, 0: overwrite it
    int unchecked;           // 1: a view's rows and samples can be counted by the unchecked taps
    float2 cs[BP_MAX_ANGLES];   // (cos phi, sin phi) of each view
    int first_view;          // index of cs[0] in the filtered stack
    int first_group;         // group of BP_ZT slices of the launch's first block
};

__device__ __forceinline__ float tap(const float* __restrict__ img, int nu, int nv, int iu, int iv) {
    return (iu >= 0 && iu < nu && iv >= 0 && iv < nv) ? __ldg(img + (size_t)iv * nu + iu) : 0.0f;
}

// A warp covers 8 x 4 columns, so that its detector samples of one view span a
// few cache lines whatever the gantry angle (a row of 32 columns spans 125
// samples at 90 degrees).  A group of voxels that misses the detector is left
// at once; one whose samples all lie inside takes them unchecked, its row
// index by adding 2^23 rounded down; only one across an edge tests every tap.
//
// The arithmetic of two voxels of a column runs in packed pairs.
//
// Bound: instruction issue (70 % of the slots) beside L1 (64 %).  3.0e9
// voxel-views (360 views of 512 x 384, 256 x 256 x 128 voxels of 2 mm, more
// than half of them beyond the detector): 4.4 ms with rows of 32 columns and
// every tap tested, 2.4 ms without, 2.26 ms in pairs.  Groups of 6 and 8 voxels
// were 2 to 4 % slower, 2 and 16 more so; five resident blocks 5 % slower and four
// 1 % slower than three with their registers.
__global__ void __launch_bounds__(BP_BX * BP_BY, 3) fdk_backproject_kernel(const BpParams p, const float* __restrict__ q,
                                                                       float* __restrict__ vol) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ix = blockIdx.x * BP_BX + (warp % (BP_BX / BP_WX)) * BP_WX + lane % BP_WX;
    const int iy = blockIdx.y * BP_BY + (warp / (BP_BX / BP_WX)) * (32 / BP_WX) + lane / BP_WX;
    const int iz0 = (p.first_group + (int)blockIdx.z) * BP_ZT;
    if (ix >= p.nx || iy >= p.ny) return;
    const float x = p.x0 + (float)ix * p.dx;
    const float y = p.y0 + (float)iy * p.dy;
    uint64_t accp[BP_ZT / 2], zp[BP_ZT / 2];
#pragma unroll
    for (int h = 0; h < BP_ZT / 2; ++h) {
        accp[h] = 0ull;
        zp[h] = pack2(bp_height(p.z0, iz0 + 2 * h, p.dz), bp_height(p.z0, iz0 + 2 * h + 1, p.dz));
    }
    const size_t view = (size_t)p.nu * p.nv;
    const float z_lo = bp_height(p.z0, iz0, p.dz), z_hi = bp_height(p.z0, iz0 + BP_ZT - 1, p.dz);
    for (int i = 0; i < p.n_ang; ++i) {
        const float cph = p.cs[i].x, sph = p.cs[i].y;
        const float depth = p.sad + x * cph + y * sph;
        // the rounded reciprocal: the approximate one (within 1 ulp) and Newton's step,
        // equal to 1 / depth for every significand (all 2^23 compared)
        float inv;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(depth));
        inv = fmaf(inv, fmaf(-depth, inv, 1.0f), inv);
        const float fu = p.sad * (x * sph - y * cph) * inv * p.inv_tau_u + p.hu;
        const float fiu = floorf(fu);
        if (fiu < -1.0f || fiu > (float)(p.nu - 1)) continue;   // the column misses the detector
        const int iu = (int)fiu;
        const float wu = fu - fiu;
        const float m = p.sad * inv;
        const float w2 = p.d_beta * (m * m);
        const float sv = m * p.inv_tau_v;                           // dv-index per mm of z
        const float* img = q + (size_t)(p.first_view + i) * view;
        const float wu0 = 1.0f - wu;
        const float v_lo = bp_row(z_lo, sv, p.hv), v_hi = bp_row(z_hi, sv, p.hv);
        if (v_hi <= -1.0f || v_lo >= (float)p.nv) continue;        // its voxels miss the detector
        if (p.unchecked && iu >= 0 && iu < p.nu - 1 && bp_rows_inside(v_lo, v_hi, p.nv)) {
            // 0x4b000000 + iv is the bit pattern of 2^23 + iv
            const uint32_t nu = (uint32_t)p.nu, first = (uint32_t)iu - 0x4b000000u * nu;
            const uint64_t svp = twice(sv), wup = twice(wu), wu0p = twice(wu0), w2p = twice(w2);
#pragma unroll
            for (int h = 0; h < BP_ZT / 2; ++h) {                     // two voxels as packed pairs
                const uint64_t fv = fma2(zp[h], svp, twice(p.hv));   // bp_row of both
                const uint64_t t = add2_down(fv, twice(8388608.0f));   // 2^23 + floor(fv)
                const uint64_t wv = fma2(add2(t, twice(-8388608.0f)), twice(-1.0f), fv);
                float2 v[4];
                const float2 tf = unpack2(t);
                {
                    const uint32_t o = __float_as_uint(tf.x) * nu + first;
                    const float *r0 = img + o, *r1 = img + (o + nu);
                    v[0].x = __ldg(r0); v[1].x = __ldg(r0 + 1); v[2].x = __ldg(r1); v[3].x = __ldg(r1 + 1);
                }
                {
                    const uint32_t o = __float_as_uint(tf.y) * nu + first;
                    const float *r0 = img + o, *r1 = img + (o + nu);
                    v[0].y = __ldg(r0); v[1].y = __ldg(r0 + 1); v[2].y = __ldg(r1); v[3].y = __ldg(r1 + 1);
                }
                const uint64_t a = fma2(wup, pack2(v[1].x, v[1].y), mul2(wu0p, pack2(v[0].x, v[0].y)));
                const uint64_t b = fma2(wup, pack2(v[3].x, v[3].y), mul2(wu0p, pack2(v[2].x, v[2].y)));
                const uint64_t wv0 = fma2(wv, twice(-1.0f), twice(1.0f));
                accp[h] = fma2(w2p, fma2(wv, b, mul2(wv0, a)), accp[h]);
            }
            continue;
        }
#pragma unroll
        for (int k = 0; k < BP_ZT; ++k) {
            // clamped two samples beyond the edges (those taps read zero)
            const float fv = fminf(fmaxf(bp_row(bp_height(p.z0, iz0 + k, p.dz), sv, p.hv), -2.0f), (float)p.nv + 1.0f);
            const float fiv = floorf(fv);
            const int iv = (int)fiv;
            const float wv = fv - fiv;
            const float v00 = tap(img, p.nu, p.nv, iu, iv), v10 = tap(img, p.nu, p.nv, iu + 1, iv);
            const float v01 = tap(img, p.nu, p.nv, iu, iv + 1), v11 = tap(img, p.nu, p.nv, iu + 1, iv + 1);
            const float s = w2 * ((1.0f - wv) * (wu0 * v00 + wu * v10) + wv * (wu0 * v01 + wu * v11));
            accp[k / 2] = add2(accp[k / 2], k & 1 ? pack2(0.0f, s) : pack2(s, 0.0f));
        }
    }
#pragma unroll
    for (int k = 0; k < BP_ZT; ++k) {
        const int iz = iz0 + k;
        const float2 a = unpack2(accp[k / 2]);
        if (iz < p.nz) {
            const size_t o = ((size_t)iz * p.ny + iy) * p.nx + ix;
            vol[o] = (p.accumulate ? vol[o] : 0.0f) + (k & 1 ? a.y : a.x);
        }
    }
}

// Line integrals -ln(max(s, floor a) / a), rounded to FP32 from the FP64
// inputs.  GB300 runs FP64 at 1/64 of the FP32 rate and the FP64 logarithm
// bound the kernel (5.2 ms for 70.8 M pixels against 0.13 ms of memory
// traffic), 0.42 ms as below: the value is formed in pairs of floats from the integer bits of
// the operands: with r = s / a brought to [sqrt(1/2), sqrt(2)) by a power of
// two, ln r = 2 atanh(t), t = (ms - ma) / (ms + ma) (difference and sum of the
// 53-bit significands, quotient with its remainder), atanh t = t (1 + c) by its
// Taylor series to t^15, c = u (1/3 + u (1/5 + u q)), u = t^2, with q alone a
// single float.
//
// Relative error of the pair, below 2^-39.5: |t| <= 0.1716, so u <= 0.0295 and
// u q <= 0.0043; q and u q carry four roundings of 2^-24 (q's last step, its
// constant, u's low part left out, the product), which u^2 <= 8.7e-4 scales to
// 4.3 x 0.0043 x 8.7e-4 x 2^-24 < 2^-39.8.  The terms left out (t^16 / 17 and on:
// 2^-44.7), and the roundings of the pairs' low parts (t, u, the outer steps, the
// sums with e ln 2: at most 2^-43 each) come to less than 2^-41.  (The largest of
// 1.8e7 values against a 113-bit logarithm: 2^-39.97, whether the reciprocal is
// rounded or off by one ulp either way.)  Where an error of 2^-38 leaves the
// rounding to FP32 open (one pixel in about 8000), and for operands that are not
// positive normal numbers, the FP64 logarithm decides: what is written is the
// FP32 rounding of the logarithm.
constexpr int LI_VIEWS = 8;       // pixels of consecutive views per thread: the air pixel's part is formed once

struct Pair {
    float h, l;
};

__device__ __forceinline__ Pair two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ Pair fast_two_sum(float a, float b) {      // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// the significand of a positive normal double as a pair in [1, 2): its first
// 24 bits, and the 29 below as an integer (units of 2^-52)
struct Significand {
    float h;
    int l;
};
constexpr float TWO_M52 = (float)(1.0 / 4503599627370496.0);

__device__ __forceinline__ Significand significand(uint64_t bits) {
    return {__uint_as_float(0x3f800000u | ((uint32_t)(bits >> 29) & 0x007fffffu)), (int)((uint32_t)bits & 0x1fffffffu)};
}

// Near a ratio of one the quotient's own rounding is all that its logarithm
// would show, so there the difference (exact) is divided instead.
__device__ __noinline__ float line_integral_64(double s, double a, double floor_rel) {
    const double v = fmax(s, floor_rel * a), x = v - a;
    return (float)(fabs(x) <= 0.5 * a ? -log1p(x / a) : -log(v / a));
}

__device__ __forceinline__ float line_integral(double s, double a, double least, double floor_rel,
                                               Significand ma) {
    const int64_t sb = __double_as_longlong(s), lb = __double_as_longlong(least);
    const int64_t vb = sb > lb ? sb : lb;                 // positive doubles order like their bits
    const int64_t ab = __double_as_longlong(a);
    const int ev = (int)(vb >> 52), ea = (int)(ab >> 52);
    if ((unsigned)(ev - 1) >= 2046u || (unsigned)(ea - 1) >= 2046u || lb <= 0) return line_integral_64(s, a, floor_rel);
    const Significand mv = significand((uint64_t)vb);
    // the power of two k that brings the ratio to [sqrt(1/2), sqrt(2)); the
    // difference mv - k ma: that of the heads is exact (a ratio within 2), that of
    // the low parts an integer below 2^31, whatever k, taken as two floats
    int e = ev - ea, dl = mv.l - ma.l;
    float k = 1.0f, unit = TWO_M52;
    if (mv.h > 1.41421354f * ma.h) { k = 2.0f; e += 1; dl -= ma.l; }
    else if (1.41421354f * mv.h < ma.h) { k = 0.5f; e -= 1; dl += mv.l; unit = 0.5f * TWO_M52; }
    const float ah = k * ma.h;
    const float d1 = (float)dl, d2 = (float)(dl - (int)d1);
    Pair d = two_sum(__fsub_rn(mv.h, ah), d1 * unit);
    d = two_sum(d.h, __fmaf_rn(d2, unit, d.l));
    Pair w = two_sum(mv.h, ah);
    w.l = __fadd_rn(w.l, __fadd_rn((float)mv.l * TWO_M52, (float)ma.l * (k * TWO_M52)));
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(w.h));
    Pair t;
    t.h = __fmul_rn(d.h, y);
    t.l = __fmul_rn(__fadd_rn(__fmaf_rn(-t.h, w.h, d.h), __fmaf_rn(-t.h, w.l, d.l)), y);
    t = fast_two_sum(t.h, t.l);
    const float uh = __fmul_rn(t.h, t.h);
    const float ul = __fmaf_rn(2.0f * t.h, t.l, __fmaf_rn(t.h, t.h, -uh));
    float q = (float)(1.0 / 15.0);
    q = __fmaf_rn(q, uh, (float)(1.0 / 13.0));
    q = __fmaf_rn(q, uh, (float)(1.0 / 11.0));
    q = __fmaf_rn(q, uh, (float)(1.0 / 9.0));
    q = __fmaf_rn(q, uh, (float)(1.0 / 7.0));
    // c = u (1/3 + u (1/5 + u q)), the two outer steps in pairs
    constexpr float C3H = (float)(1.0 / 3.0), C3L = (float)(1.0 / 3.0 - (double)C3H);
    constexpr float C5H = (float)(1.0 / 5.0), C5L = (float)(1.0 / 5.0 - (double)C5H);
    Pair p = fast_two_sum(C5H, __fmul_rn(uh, q));
    p.l = __fadd_rn(p.l, C5L);
    const float vh = __fmul_rn(uh, p.h);
    const float vl = __fadd_rn(__fmaf_rn(uh, p.h, -vh), __fmaf_rn(uh, p.l, __fmul_rn(ul, p.h)));
    p = fast_two_sum(C3H, vh);
    p.l = __fadd_rn(p.l, __fadd_rn(vl, C3L));
    const float ch = __fmul_rn(uh, p.h);
    const float cl = __fadd_rn(__fmaf_rn(uh, p.h, -ch), __fmaf_rn(uh, p.l, __fmul_rn(ul, p.h)));
    // ln r = 2 (t + t c)
    const float bh = __fmul_rn(t.h, ch);
    const float bl = __fadd_rn(__fmaf_rn(t.h, ch, -bh), __fmaf_rn(t.h, cl, __fmul_rn(t.l, ch)));
    Pair g = fast_two_sum(t.h, bh);
    g.l = __fadd_rn(g.l, __fadd_rn(t.l, bl));
    // + e ln 2: e times the 12-bit head is exact
    const float fe = (float)e;
    constexpr double LN2 = 0.69314718055994530942;
    constexpr float L1 = (float)(2839.0 / 4096.0), L2 = (float)(LN2 - 2839.0 / 4096.0);
    constexpr float L3 = (float)(LN2 - 2839.0 / 4096.0 - (double)L2);
    const float mh = __fmul_rn(fe, L2);
    const Pair f = two_sum(__fmul_rn(fe, L1), 2.0f * g.h);
    const Pair m = two_sum(f.h, mh);
    const float lo = __fadd_rn(__fadd_rn(f.l, m.l), __fmaf_rn(2.0f, g.l, __fmaf_rn(fe, L3, __fmaf_rn(fe, L2, -mh))));
    const Pair r = fast_two_sum(m.h, lo);
    const float err = fabsf(r.h) * (float)(1.0 / 274877906944.0);            // 2^-38
    if (__fadd_rn(r.h, __fadd_rn(r.l, err)) != r.h || __fadd_rn(r.h, __fsub_rn(r.l, err)) != r.h)
        return line_integral_64(s, a, floor_rel);
    return -r.h;
}

__global__ void __launch_bounds__(256) line_integral_kernel(const double* __restrict__ s, const double* __restrict__ a,
                                                           int64_t n_views, int64_t n, double floor_rel,
                                                           float* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double i0 = a[i], least = floor_rel * i0;
    const Significand ma = significand((uint64_t)__double_as_longlong(i0));
    const int64_t v0 = (int64_t)blockIdx.y * LI_VIEWS;
#pragma unroll
    for (int k = 0; k < LI_VIEWS; ++k)
        if (v0 + k < n_views) out[(v0 + k) * n + i] = line_integral(s[(v0 + k) * n + i], i0, least, floor_rel, ma);
}

bool geometry_valid(const gdrr_fdk_geometry* g) {
    return g && g->sad_mm > 0 && g->sdd_mm > g->sad_mm && g->nu > 0 && g->nv > 0 && g->du_mm > 0 && g->dv_mm > 0
           && g->nx > 0 && g->ny > 0 && g->nz > 0 && g->dx_mm > 0 && g->dy_mm > 0 && g->dz_mm > 0
           && std::isfinite(g->sad_mm) && std::isfinite(g->sdd_mm);
}

}  // namespace
}  // namespace gdrr

extern "C" GDRR_API int gdrr_line_integrals_views(const double* signal_dev, const double* air_dev, int64_t n_views,
                                                  int64_t n, double floor_rel, float* out_dev, void* cuda_stream) {
    if (n < 0 || n_views < 0 || (n > 0 && n_views > 0 && (!signal_dev || !air_dev || !out_dev)) || !(floor_rel > 0.0)
        || !(floor_rel < 1.0))
        return GDRR_ERR_INVALID_ARG;
    if (n == 0 || n_views == 0) return GDRR_OK;
    if (n_views > 65535 * (int64_t)gdrr::LI_VIEWS) return GDRR_ERR_UNSUPPORTED;
    const int block = 256;
    const dim3 grid((unsigned)((n + block - 1) / block), (unsigned)((n_views + gdrr::LI_VIEWS - 1) / gdrr::LI_VIEWS));
    gdrr::line_integral_kernel<<<grid, block, 0, (cudaStream_t)cuda_stream>>>(signal_dev, air_dev, n_views, n, floor_rel,
                                                                             out_dev);
    return cudaGetLastError() == cudaSuccess ? GDRR_OK : GDRR_ERR_CUDA;
}

extern "C" GDRR_API int gdrr_line_integrals(const double* signal_dev, const double* air_dev, int64_t n,
                                            double floor_rel, float* out_dev, void* cuda_stream) {
    return gdrr_line_integrals_views(signal_dev, air_dev, 1, n, floor_rel, out_dev, cuda_stream);
}

extern "C" GDRR_API int gdrr_fdk_filter(const gdrr_fdk_geometry* g, int32_t n_proj, const float* proj_dev,
                                        float* filtered_dev, void* cuda_stream) {
    if (!gdrr::geometry_valid(g) || n_proj < 0 || (n_proj > 0 && (!proj_dev || !filtered_dev)))
        return GDRR_ERR_INVALID_ARG;
    if (g->nu > gdrr::FILTER_MAX_NU || g->nv > 65535 || n_proj > 65535) return GDRR_ERR_UNSUPPORTED;
    if (n_proj == 0) return GDRR_OK;
    gdrr::FilterParams p;
    const double mag = g->sad_mm / g->sdd_mm;
    p.nu = g->nu; p.nv = g->nv;
    p.mag_du = (float)(g->du_mm * mag);
    p.mag_dv = (float)(g->dv_mm * mag);
    p.sad = (float)g->sad_mm;
    p.scale = (float)(0.5 / (g->du_mm * mag));
    const int64_t n_rows = (int64_t)g->nv * n_proj, n = n_rows * g->nu;
    const bool apart = std::less_equal<const float*>()(proj_dev + n, filtered_dev) ||
                       std::less_equal<const float*>()(filtered_dev + n, proj_dev);
    int dev = 0, n_sm = 1;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return GDRR_ERR_CUDA;
    const gdrr::FilterShape f = gdrr::filter_shape(g->nu, n_rows, n_sm, apart);
    if (gdrr::allow_smem(gdrr::fdk_filter_kernel, gdrr::filter_smem_most()) != cudaSuccess) return GDRR_ERR_CUDA;
    const dim3 grid((unsigned)((n_rows + f.rows - 1) / f.rows), (unsigned)f.parts);
    gdrr::fdk_filter_kernel<<<grid, gdrr::FILTER_BLOCK, gdrr::filter_smem(f), (cudaStream_t)cuda_stream>>>(
        p, f, n_rows, proj_dev, filtered_dev);
    return cudaGetLastError() == cudaSuccess ? GDRR_OK : GDRR_ERR_CUDA;
}

extern "C" GDRR_API int gdrr_fdk_backproject(const gdrr_fdk_geometry* g, int32_t n_proj, const double* angles_rad,
                                             double d_beta, const float* filtered_dev, float* volume_dev,
                                             int32_t accumulate, void* cuda_stream) {
    if (!gdrr::geometry_valid(g) || n_proj < 0 || !volume_dev || (n_proj > 0 && (!angles_rad || !filtered_dev))
        || !std::isfinite(d_beta) || (accumulate != 0 && accumulate != 1))
        return GDRR_ERR_INVALID_ARG;
    for (int i = 0; i < n_proj; ++i)
        if (!std::isfinite(angles_rad[i])) return GDRR_ERR_INVALID_ARG;
    // every voxel must lie on the source's side of the isocentre plane at
    // every angle (depth > 0): the grid's half-diagonal stays below SAD
    const double hx = 0.5 * g->nx * g->dx_mm, hy = 0.5 * g->ny * g->dy_mm;
    if (!(std::sqrt(hx * hx + hy * hy) < g->sad_mm)) return GDRR_ERR_INVALID_ARG;
    if ((int64_t)g->ny > 65535 * (int64_t)gdrr::BP_BY) return GDRR_ERR_UNSUPPORTED;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const double mag = g->sad_mm / g->sdd_mm;
    gdrr::BpParams p;
    p.nx = g->nx; p.ny = g->ny; p.nz = g->nz; p.nu = g->nu; p.nv = g->nv;
    p.x0 = (float)((0.5 - 0.5 * g->nx) * g->dx_mm);
    p.y0 = (float)((0.5 - 0.5 * g->ny) * g->dy_mm);
    p.z0 = (float)((0.5 - 0.5 * g->nz) * g->dz_mm);
    p.dx = (float)g->dx_mm; p.dy = (float)g->dy_mm; p.dz = (float)g->dz_mm;
    p.sad = (float)g->sad_mm;
    p.inv_tau_u = (float)(1.0 / (g->du_mm * mag));
    p.inv_tau_v = (float)(1.0 / (g->dv_mm * mag));
    p.hu = (float)(0.5 * g->nu - 0.5);
    p.hv = (float)(0.5 * g->nv - 0.5);
    p.d_beta = (float)d_beta;
    p.unchecked = g->nv < (1 << 22) && (int64_t)g->nu * g->nv < ((int64_t)1 << 31) ? 1 : 0;
    const int block = gdrr::BP_BX * gdrr::BP_BY;
    // (a launch has at most 65535 blocks in z: taller volumes take several)
    const int groups = (g->nz - 1) / gdrr::BP_ZT + 1;
    if (n_proj == 0 && !accumulate) {
        if (cudaMemsetAsync(volume_dev, 0, sizeof(float) * (size_t)g->nx * g->ny * g->nz, s) != cudaSuccess)
            return GDRR_ERR_CUDA;
        return GDRR_OK;
    }
    for (int first = 0; first < n_proj; first += gdrr::BP_MAX_ANGLES) {
        const int n = std::min(gdrr::BP_MAX_ANGLES, n_proj - first);
        p.n_ang = n;
        p.first_view = first;
        p.accumulate = (first > 0 || accumulate) ? 1 : 0;
        for (int i = 0; i < n; ++i)
            p.cs[i] = make_float2((float)std::cos(angles_rad[first + i]), (float)std::sin(angles_rad[first + i]));
        for (p.first_group = 0; p.first_group < groups; p.first_group += 65535) {
            const dim3 grid((unsigned)((g->nx + gdrr::BP_BX - 1) / gdrr::BP_BX),
                            (unsigned)((g->ny + gdrr::BP_BY - 1) / gdrr::BP_BY),
                            (unsigned)std::min(65535, groups - p.first_group));
            gdrr::fdk_backproject_kernel<<<grid, block, 0, s>>>(p, filtered_dev, volume_dev);
            if (cudaGetLastError() != cudaSuccess) return GDRR_ERR_CUDA;
        }
    }
    return GDRR_OK;
}
