// Monte Carlo photon transport, Section 2.4 of the paper, for sm_103a.
//
// The grid is persistent: warps claim chunks of histories from a global
// counter, and each warp keeps a pool of photons in shared memory from which
// it runs the common event (a Woodcock free flight that ends in a virtual
// collision) and each of the rare, long ones (corner gathers, Rayleigh /
// Compton sampling, the detector tally and the start of a new history) on
// whole warps (mc_warp_kernel).  Runs with event records keep one photon per
// lane (mc_kernel).  Tallies are int64 fixed point (2^-24 keV), summed with
// integer atomics, so the result does not depend on which lane ran which
// history, when, or in which order.
//
// Data layout: one 8-byte record {density bits, material index} per voxel,
// in bricks of 4 x 2 x 2 voxels (one 128-byte cache line each), so each
// trilinear corner is a single 8-byte gather and the eight corners of a cell
// touch about 2.8 distinct lines instead of about 4.3 for a row-major layout;
// the energy-dependent coefficients of a photon live in shared memory, indexed
// by material.
//
// Most tentative collisions of Woodcock tracking are virtual (over 90 % in a
// torso, whose majorant is set by dense bone).  Before the eight corner
// gathers, a tentative collision is compared with a bound on mu over the
// macro cell that holds the corners (a small table: the largest density of
// each material per cell); above it the collision is virtual whatever the
// corners hold, and the gathers are skipped.  The bound never falls below the
// mu the gathers give, so every decision, draw and tally is the one plain
// Woodcock tracking makes.  A flight that passes the test waits, like the rare
// events, for a service of the warp, where its gathers run together with those
// of the warp's other waiting photons.
//
// Local majorants (an option, LM): the macro-cell bounds themselves serve as a
// piecewise-constant majorant.  A flight draws its optical depth tau = -ln xi
// and spends it cell by cell along the ray (a cell of bound b crossed whole
// costs b times its chord); where it runs out, tau / b into the cell, lies the
// tentative collision, real with probability mu / b (the same ordinate test,
// t = xi' b against the mixture).  Cheap cell crossings replace most of the
// flights (about 46 per history in the torso with the global majorant, 4 to 6
// with 16 to 32 mm cells); the tentative collisions wait for the service
// batch, where the gathers, the decision and the next flight's Philox block
// run on the warp's waiting lanes together.
//
// Arithmetic contract.  This file is compiled with -fmad=false: every FP32
// operation below is one IEEE-rounded operation, evaluated in the order
// written (divide and square root are the correctly rounded ones).  The only
// transcendental is the logarithm of the free-flight length, computed by the
// atanh series in gd_logf below.  Together with the counter-based random
// streams this makes a history's result a function of (seed, angle index,
// history id) alone.
//
// Readings of points the paper leaves open:
//  * random numbers: Philox4x32-10 (Salmon et al., SC'11), key = seed,
//    counter = (block, angle index, history id lo, hi), one whole block per
//    draw site; uniforms are ((word >> 8) + 1) * 2^-24 in (0, 1];
//  * source: detector pixel from the fluence map w(u) and channel from the
//    spectrum phi(E), each by inverse CDF; uniform point inside the pixel;
//  * material at an off-centre point: trilinear mixture of the eight corner
//    voxels, mu_k(x, E) = sum_c w_c rho_c mu_hat_k(m_c, E) (the density
//    interpolation of Section 2.4, the same field the ray tracer of Section
//    2.3 integrates); the total decides real versus virtual, then one uniform
//    picks Rayleigh, Compton or photoelectric in that order;
//  * field: clamp to edge inside the voxel box, vacuum outside;
//  * Woodcock majorant mu_max(E): largest mu over materials at their largest
//    density, the larger of the two bracketing energy nodes;
//  * Compton: free-electron Klein-Nishina by Kahn's rejection method;
//    Rayleigh: Thomson (1 + cos^2) by rejection; azimuth from a point of the
//    unit disc;
//  * tally: rint(r(E) * 2^24) into the primary counter when the photon never
//    scattered, else the scatter counter (Section 2.4).
#include <algorithm>

#include "gdrr_internal.cuh"
#include "transport_rules.h"

namespace gdrr {
namespace {

// The macro-cell bound is raised by 2^-10, far above the rounding of the
// eight-corner mixture (eleven FP32 operations on the way to mu, each within
// 2^-24 relative), so mu as the kernel computes it never exceeds it.
constexpr float CELL_MARGIN = 1.0009765625f;

// Rejection samplers stop rejecting once their history has drawn this many
// Philox blocks and keep the candidate in hand (the azimuth takes phi = 0).
// A legal history stays far below it (at most max_steps flights plus a few
// tries per interaction, and every sampler accepts with probability at
// least 1/2); it bounds the loops for inputs that are not finite.
constexpr uint32_t MAX_BLOCKS = 1u << 24;

constexpr unsigned FULL = 0xffffffffu;

// Ten Philox rounds with the round keys k_r = key + r (0x9E3779B9, 0xBB67AE85)
// precomputed on the host (they depend only on the seed), so each round is
// two wide multiplies and two three-input XORs with a constant-bank operand.
// Each product is one 32 x 32 -> 64-bit multiply whose halves are the round's
// high and low words (0.6 % fewer instructions per flight than a low
// multiply beside a separate high multiply).
__device__ __forceinline__ void philox4x32_10(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& c3,
                                              const RoundKeys& rk) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ rk.k0[r];
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ rk.k1[r];
        c0 = n0; c1 = (uint32_t)p1; c2 = n2; c3 = (uint32_t)p0;
    }
}

// The random stream of one history: Philox blocks with counter (k, angle
// index, history id lo, hi), k = 0, 1, 2, ...; every draw site takes the next
// whole block (source, each free flight, each rejection attempt), so the
// Philox rounds of a free flight run on all lanes of a warp together.
struct Stream {
    uint32_t angle, hlo, hhi, blk;

    __device__ __forceinline__ void init(uint32_t angle_index, uint64_t hid) {
        angle = angle_index; hlo = (uint32_t)hid; hhi = (uint32_t)(hid >> 32);
        blk = 0;
    }
    __device__ __forceinline__ uint4 block(const RoundKeys& rk) {
        uint32_t c0 = blk, c1 = angle, c2 = hlo, c3 = hhi;
        philox4x32_10(c0, c1, c2, c3, rk);
        ++blk;
        return make_uint4(c0, c1, c2, c3);
    }
};

// Uniform on (0, 1]: the top 24 bits plus one, times 2^-24 (exact in FP32).
__device__ __forceinline__ float uniform(uint32_t w) {
    return (float)((w >> 8) + 1u) * (float)(1.0 / 16777216.0);
}

// ln(x), x a positive normal float: x = m 2^e, m in [sqrt(1/2), sqrt(2)),
// ln m = 2 atanh(s), s = (m - 1)/(m + 1), by the Taylor series of atanh to
// s^11 (|s| <= 0.1716, remainder below 2^-30), ln 2 split into a 12-bit head
// (exact products with e) and a tail.
__device__ __forceinline__ float gd_logf(float x) {
    uint32_t u = __float_as_uint(x);
    int e = (int)((u >> 23) & 0xffu) - 127;
    u = (u & 0x007fffffu) | 0x3f800000u;
    if (u > 0x3fb504f3u) {
        u -= 0x00800000u;
        e += 1;
    }
    const float m = __uint_as_float(u);
    const float s = (m - 1.0f) / (m + 1.0f);
    const float s2 = s * s;
    const float poly = (float)(1.0 / 3.0) + s2 * ((float)(1.0 / 5.0) + s2 * ((float)(1.0 / 7.0)
                     + s2 * ((float)(1.0 / 9.0) + s2 * (float)(1.0 / 11.0))));
    const float lm = 2.0f * s + (2.0f * s) * (s2 * poly);
    const float fe = (float)e;
    return fe * (float)(2839.0 / 4096.0) + (fe * (float)(0.69314718055994530942 - 2839.0 / 4096.0) + lm);
}

// n / d for the logarithm's arguments (n = m - 1, d = m + 1, m in
// [sqrt(1/2), sqrt(2))): the quotient from an approximate reciprocal and
// Markstein's residual correction (P. Markstein, IBM J. Res. Dev. 34, 1990).
// Equal to the correctly rounded quotient for every m of a 24-bit uniform (all
// 2^24 compared), without the general division's range test and branch.
__device__ __forceinline__ float log_quotient(float n, float d) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d));
    const float q = __fmul_rn(n, y);
    return __fmaf_rn(__fmaf_rn(-d, q, n), y, q);
}

// gd_logf(k 2^-24) for an integer 1 <= k <= 2^24: the same series on the same
// m and e, which one addition separates (it carries into the exponent exactly
// when the mantissa exceeds sqrt(2)'s).
__device__ __forceinline__ float log_uniform(uint32_t k) {
    constexpr uint32_t CARRY = 0x00800000u - 0x003504f4u;
    const uint32_t t = __float_as_uint((float)k) + CARRY;
    const float fe = __uint_as_float(0x4b000000u | (t >> 23)) - 8388759.0f;     // (t >> 23) - 127 - 24
    const float m = __uint_as_float((t & 0x007fffffu) + (0x3f800000u - CARRY));
    const float s = log_quotient(m - 1.0f, m + 1.0f);
    const float s2 = s * s;
    const float poly = (float)(1.0 / 3.0) + s2 * ((float)(1.0 / 5.0) + s2 * ((float)(1.0 / 7.0)
                     + s2 * ((float)(1.0 / 9.0) + s2 * (float)(1.0 / 11.0))));
    const float lm = 2.0f * s + (2.0f * s) * (s2 * poly);
    return fe * (float)(2839.0 / 4096.0) + (fe * (float)(0.69314718055994530942 - 2839.0 / 4096.0) + lm);
}

// Inverse-CDF search in integers.  A uniform is xi = k 2^-24 with k the top
// 24 bits of its word plus one, and xi <= cdf[j] holds exactly when
// k <= floor(cdf[j] 2^24) = kcdf[j]; the smallest such j is the sample.  The
// guide table gives a start, two short scans finish.
__device__ __forceinline__ int cdf_search(const uint32_t* __restrict__ kcdf, const int* __restrict__ guide,
                                          int n_guide, uint32_t w) {
    const uint32_t k = (w >> 8) + 1u;
    int gi = (int)(((uint64_t)k * (uint64_t)n_guide) >> 24);
    gi = gi > n_guide - 1 ? n_guide - 1 : gi;
    int j = __ldg(guide + gi);
    while (j > 0 && k <= __ldg(kcdf + j - 1)) --j;
    while (k > __ldg(kcdf + j)) ++j;
    return j;
}

__device__ __forceinline__ void interp_index(float e, float e0, float inv_de, int n, int& i, float& f) {
    float fi = (e - e0) * inv_de;
    if (fi < 0.0f) fi = 0.0f;
    if (fi > (float)(n - 1)) fi = (float)(n - 1);
    int ie = (int)fi;
    if (ie > n - 2) ie = n - 2;
    i = ie;
    f = fi - (float)ie;
}

__device__ __forceinline__ float response(const McParams& P, float e) {
    int ir; float f;
    interp_index(e, P.r0, P.inv_dr, P.n_r, ir, f);
    const float a = __ldg(P.resp + ir), b = __ldg(P.resp + ir + 1);
    return a + f * (b - a);
}

__device__ __forceinline__ void azimuth(Stream& rs, const RoundKeys& rk, float& cp, float& sp) {
    while (rs.blk < MAX_BLOCKS) {
        const uint4 w = rs.block(rk);
        const float a = 2.0f * uniform(w.x) - 1.0f;
        const float b = 2.0f * uniform(w.y) - 1.0f;
        const float r2 = a * a + b * b;
        if (r2 <= 1.0f && r2 > 0.0f) {
            const float inv = 1.0f / r2;
            cp = (a * a - b * b) * inv;
            sp = 2.0f * a * b * inv;
            return;
        }
    }
    cp = 1.0f;
    sp = 0.0f;
}

__device__ __forceinline__ void rotate(float& u, float& v, float& w, float ct, float cp, float sp) {
    const float st2 = 1.0f - ct * ct;
    const float st = st2 > 0.0f ? sqrtf(st2) : 0.0f;
    float nu_, nv_, nw_;
    if (w < (float)0.99999 && w > (float)-0.99999) {
        const float t = sqrtf(1.0f - w * w);
        const float sti = st / t;
        nu_ = u * ct + sti * (u * w * cp - v * sp);
        nv_ = v * ct + sti * (v * w * cp + u * sp);
        nw_ = w * ct - st * t * cp;
    } else {
        nu_ = st * cp;
        nv_ = st * sp;
        nw_ = w > 0.0f ? ct : -ct;
    }
    const float il = 1.0f / sqrtf(nu_ * nu_ + nv_ * nv_ + nw_ * nw_);
    u = nu_ * il;
    v = nv_ * il;
    w = nw_ * il;
}

// Rayleigh polar angle with the form factor of material m at energy e: the
// density of s = x^2 is F^2(s), linear in s between the table's nodes, so
// its cumulative is the trapezoid sum on the nodes and quadratic within an
// interval.  s is drawn on [0, s_max], s_max = (e / hc)^2, by inverse CDF
// (binary search for the interval, the root of the quadratic within it),
// cos = 1 - 2 s / s_max, and accepted with (1 + cos^2) / 2.  One block per
// attempt: word 0 draws s, word 1 the acceptance.
__device__ __forceinline__ float rayleigh_ff(Stream& rs, const McParams& P, float e, int m) {
    const float* __restrict__ S = P.ff_s;
    const float* __restrict__ A = P.ff_a + (size_t)m * P.n_ff;
    const float* __restrict__ G = P.ff_g + (size_t)m * P.n_ff;
    const float xmax = e * P.inv_hc;
    const float smax = xmax * xmax;
    int j = (int)(xmax * P.ff_idx);
    if (j > P.n_ff - 2) j = P.n_ff - 2;
    const float sj = __ldg(S + j), sj1 = __ldg(S + j + 1);
    const float gj = __ldg(G + j), gj1 = __ldg(G + j + 1);
    const float hj = sj1 - sj;
    const float tj = smax - sj;
    const float amax = __ldg(A + j) + tj * (gj + (gj1 - gj) * tj / (2.0f * hj));
    for (;;) {
        const uint4 w = rs.block(P.rk);
        const float target = uniform(w.x) * amax;
        int lo = 1, hi = j + 1;        // smallest k in [1, j+1] with A[k] >= target
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(A + mid) >= target) hi = mid; else lo = mid + 1;
        }
        const float s0 = __ldg(S + lo - 1);
        const float h = __ldg(S + lo) - s0;
        const float g0 = __ldg(G + lo - 1), g1 = __ldg(G + lo);
        const float D = target - __ldg(A + lo - 1);
        float q = g0 * g0 + 2.0f * (g1 - g0) * D / h;
        if (q < 0.0f) q = 0.0f;
        float s = s0 + 2.0f * D / (g0 + sqrtf(q));
        if (s > smax) s = smax;
        float ct = 1.0f - 2.0f * s / smax;
        if (!(ct >= -1.0f)) ct = -1.0f;
        if (2.0f * uniform(w.y) <= 1.0f + ct * ct || rs.blk >= MAX_BLOCKS) return ct;
    }
}

// The polar angle of a Rayleigh or Compton event, in one rejection loop for
// both kinds: each attempt draws the history's next block and applies the
// event's own test, so a warp serving both kinds runs one Philox per attempt
// instead of one per kind.
//  * Rayleigh (Thomson law): mu = 2 a - 1 accepted when 2 b <= 1 + mu^2.
//  * Compton (Klein-Nishina, Kahn's method): with alpha = E / 511 keV, branch
//    r1 <= (1 + 2 alpha) / (9 + 2 alpha) takes x = 1 + 2 alpha r2 and accepts
//    when r3 <= 4 (x - 1) / x^2; else x = (1 + 2 alpha) / (1 + 2 alpha r2),
//    accepted when r3 <= (cos^2 + 1/x) / 2; cos = 1 - (x - 1) / alpha and
//    E' = E / x.
// A history that has drawn MAX_BLOCKS blocks keeps its candidate.
__device__ __forceinline__ void polar(Stream& rs, const RoundKeys& rk, bool ray, float e, float& ct_out,
                                      float& e_out) {
    const float alpha = e * (float)(1.0 / 510.99895);
    const float ialpha = (float)510.99895 / e;
    const float ta = 2.0f * alpha;
    const float branch = (1.0f + ta) / (9.0f + ta);
    float x = 1.0f, mu = 1.0f;
    for (;;) {
        const uint4 w = rs.block(rk);
        bool done;
        if (ray) {
            const float a = uniform(w.x);
            const float b = uniform(w.y);
            mu = 2.0f * a - 1.0f;
            done = 2.0f * b <= 1.0f + mu * mu || rs.blk >= MAX_BLOCKS;
        } else {
            const float r1 = uniform(w.x);
            const float r2 = uniform(w.y);
            const float r3 = uniform(w.z);
            const bool low = r1 <= branch;
            const float xa = 1.0f + ta * r2;
            const float quot = (low ? 4.0f * (xa - 1.0f) : 1.0f + ta) / (low ? xa * xa : xa);   // one division for both
            if (low) {
                x = xa;
                done = r3 <= quot;
            } else {
                x = quot;
                const float c = 1.0f - (x - 1.0f) * ialpha;
                done = r3 <= 0.5f * (c * c + 1.0f / x);
            }
            done = done || rs.blk >= MAX_BLOCKS;      // keep the last candidate
        }
        if (done) break;
    }
    if (ray) {
        ct_out = mu;
        e_out = e;
    } else {
        ct_out = 1.0f - (x - 1.0f) * ialpha;
        e_out = e / x;
    }
}

// The eight corners of a trilinear cell: weight times density, and material.
__device__ __forceinline__ void corners(const McParams& P, float px, float py, float pz, float (&a)[8], int (&mc)[8]) {
    const float fx = (px - P.lo[0]) * P.ivox[0] - 0.5f;
    const float fy = (py - P.lo[1]) * P.ivox[1] - 0.5f;
    const float fz = (pz - P.lo[2]) * P.ivox[2] - 0.5f;
    const int gx = (int)floorf(fx), gy = (int)floorf(fy), gz = (int)floorf(fz);
    const float tx = fx - (float)gx, ty = fy - (float)gy, tz = fz - (float)gz;
    // inside the box f lies in [-1/2, n - 1/2], so g in [-1, n - 1]: the
    // lower corner clamps only from below, the upper only from above
    const int x0 = max(gx, 0), x1 = min(gx + 1, P.nx - 1);
    const int y0 = max(gy, 0), y1 = min(gy + 1, P.ny - 1);
    const int z0 = max(gz, 0), z1 = min(gz + 1, P.nz - 1);
    const float wx0 = 1.0f - tx, wy0 = 1.0f - ty, wz0 = 1.0f - tz;
    const float wxy[4] = {wx0 * wy0, tx * wy0, wx0 * ty, tx * ty};
    const int bx[2] = {brick_x(x0), brick_x(x1)};
    const int by[2] = {brick_y(y0, P.bsy), brick_y(y1, P.bsy)};
    const int bz[2] = {brick_z(z0, P.bsz), brick_z(z1, P.bsz)};
    const int rows[4] = {by[0] + bz[0], by[1] + bz[0], by[0] + bz[1], by[1] + bz[1]};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int v = rows[c >> 1] + bx[c & 1];
        const uint2 vx = __ldg(P.vox + v);
        a[c] = (wxy[c & 3] * ((c >> 2) ? tz : wz0)) * __uint_as_float(vx.x);
        mc[c] = (int)vx.y;
    }
}

enum : uint32_t { OUT_PRIMARY = 0, OUT_SCATTER = 1, OUT_PHOTO = 2, OUT_CUTOFF = 3, OUT_MISS = 4, OUT_STEP_LIMIT = 5 };

// Lane states.  A lane whose history needs an interaction, a tally or a new
// history waits in one of the non-FLY states until enough lanes of its warp
// wait too; the warp then serves them together, which keeps the expensive
// rare branches from running with one or two active lanes.
enum : int { S_DEAD = 0, S_FLY = 1, S_RAY = 2, S_COMP = 3, S_ESC = 4, S_GATHER = 5 };

// What a local-majorant lane needs before it flies on (LM): a new flight
// (Philox block and optical depth), the reciprocal of a new direction, the
// cell of a new history's entry point.
enum : uint32_t { LM_DRAW = 1u, LM_DIR = 2u, LM_CELL = 4u, LM_ALL = 7u };

// Where a history's events are counted: block-shared counters (GDRR_NSTATS,
// flushed to the stats array at exit), or a mask of the events of one service
// that the warp then counts by ballot.
struct SharedCounts {
    unsigned long long* c;
    __device__ __forceinline__ void add(int k) { atomicAdd(c + k, 1ull); }
};
struct EventMask {
    uint32_t m;
    __device__ __forceinline__ void add(int k) { m |= 1u << k; }
    __device__ __forceinline__ bool has(int k) const { return (m >> k) & 1u; }
};

// GEN: the general kernel, which honours the nearest-voxel and scatter-filter
// options; the default kernel (GEN = false) carries neither.  LM: free flights
// with local majorants instead of the global one.
template <int NM, bool REC, bool GEN, bool LM = false>
struct Lane {
    float px, py, pz, dx, dy, dz, e;
    float mumax, inv_mumax;
    int state, scattered, job;
    uint32_t nsteps;
    uint32_t n_int;      // Compton interactions (low 16 bits) and Rayleigh (high 16 bits)
    int m_ray;           // material of the pending form-factor Rayleigh event (GEN)
    // thread totals of free flights, virtual collisions and cell-decided
    // virtual collisions.  Without GEN they are added once per history at its
    // end (flights = nsteps; cell-decided = flights that neither gathered nor
    // left the box), so the common free flight carries no counter updates.
    uint32_t c_steps, c_virt, c_skip;
    uint32_t ngath;      // flights of the current history that gathered corners (not GEN)
    bool defer_e;        // start / interact leave the energy tables to the caller
    bool need_e;         // ... which must then call set_energy(P, e) before the next flight
    float tg;            // t = xi mu_max of a flight waiting for its corner gathers
                         // (LM: xi until the flight's cell is known, then xi b)
    uint32_t wz;         // that flight block's third word (GEN: form-factor material pick)
    // LM: the flight's remaining optical depth, the direction's reciprocals,
    // the cell of the position, what the lane needs next (LM_*) and the
    // thread's count of cell crossings
    float tau, idx, idy, idz;
    int cx, cy, cz;
    uint32_t lm_need, c_cross;
    Stream rs;
    // per-thread coefficient tables in shared memory: coef[k][m][tid],
    // k = 0 total, 1 Rayleigh, 2 Compton (photoelectric is the remainder)
    float* coef;
    int stride;          // blockDim.x
    const float* tot;    // where gather() reads the totals: coef's, or a pool slot's
    int tot_stride;
    // event record (REC only)
    uint64_t gidx;
    uint32_t r_virt, r_ray, r_comp, r_first, r_raymat;
    float r_esrc;
    double r_dep;

    __device__ __forceinline__ float& cf(int k, int m) { return coef[(k * NM + m) * stride]; }
    __device__ __forceinline__ float total(int m) const { return tot[m * tot_stride]; }

    // Largest total mu at the lane's energy over a macro cell's voxels: the
    // cell's per-material maximum densities times the lane's coefficients.
    // Every corner's term rho_c mu_m(E) is at most this, and the trilinear
    // weights sum to one, so the mixture mu is at most it too.
    __device__ __forceinline__ float cell_bound(const McParams& P, int cell) {
        const float* r = P.cells + (ptrdiff_t)cell * NM;
        float b;
        if constexpr (NM == 2) {
            const float2 v = __ldg(reinterpret_cast<const float2*>(r));
            b = fmaxf(v.x * cf(0, 0), v.y * cf(0, 1));
        } else {
            b = 0.0f;
#pragma unroll
            for (int q = 0; q < NM; q += 4) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(r + q));
                b = fmaxf(b, fmaxf(fmaxf(v.x * cf(0, q), v.y * cf(0, q + 1)),
                                   fmaxf(v.z * cf(0, q + 2), v.w * cf(0, q + 3))));
            }
        }
        return b * CELL_MARGIN;
    }

    __device__ __forceinline__ void set_energy(const McParams& P, float en) {
        e = en;
        int ie; float f;
        interp_index(en, P.e0, P.inv_de, P.n_e, ie, f);
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            float r = 0.0f, c = 0.0f, t = 0.0f;
            if (m < P.n_mat) {
                const float* tb = P.tab + (size_t)m * 3 * P.n_e;
                const float r0 = __ldg(tb + ie), r1 = __ldg(tb + ie + 1);
                const float c0 = __ldg(tb + P.n_e + ie), c1 = __ldg(tb + P.n_e + ie + 1);
                const float p0 = __ldg(tb + 2 * P.n_e + ie), p1 = __ldg(tb + 2 * P.n_e + ie + 1);
                r = r0 + f * (r1 - r0);
                c = c0 + f * (c1 - c0);
                const float p = p0 + f * (p1 - p0);
                t = (r + c) + p;
            }
            cf(0, m) = t;
            cf(1, m) = r;
            cf(2, m) = c;
        }
        const float a = __ldg(P.major + ie), b = __ldg(P.major + ie + 1);
        mumax = a > b ? a : b;
        inv_mumax = 1.0f / mumax;
    }

    // a history ended; esc: its last flight left the box
    __device__ __forceinline__ void end_counts(uint32_t esc) {
        if (GEN) return;
        if (LM) {                    // no cell test: every virtual collision gathered
            c_steps += nsteps;
            return;
        }
        const uint32_t skipped = nsteps - ngath - esc;
        c_steps += nsteps;
        c_skip += skipped;
        c_virt += skipped;
    }

    __device__ __forceinline__ void record(const McParams& P, uint32_t outcome, int pixel, uint32_t photo) {
        if (!REC) return;
        gdrr_history_record r;
        r.n_steps = nsteps; r.n_virtual = r_virt; r.n_rayleigh = r_ray; r.n_compton = r_comp;
        r.n_photo = photo; r.outcome = outcome; r.rng_blocks = rs.blk; r.first_interaction = r_first;
        r.pixel = pixel; r.e_source = r_esrc; r.e_final = e; r.ray_material = r_raymat; r.e_deposited = r_dep;
        P.records[gidx] = r;
    }

    // Straight line from the box surface (or the source) to the imager
    // plane; tally r(E) at the pixel it meets (Section 2.4).  A lane that
    // left the box in a free flight first moves from its last position inside
    // to the box surface along its direction.
    template <class CNT>
    __device__ __forceinline__ void escape(const McParams& P, CNT& cnt, bool from_inside) {
        if (from_inside) move_to_box_exit(P);
        const Job& J = P.jobs[job];
        const float n0 = J.f.n[0], n1 = J.f.n[1], n2 = J.f.n[2];
        const float dn = dx * n0 + dy * n1 + dz * n2;
        uint32_t outcome = OUT_MISS;
        int pixel = -1;
        if (dn > 0.0f) {
            const float P0 = J.f.P[0], P1 = J.f.P[1], P2 = J.f.P[2];
            const float num = (P0 - px) * n0 + (P1 - py) * n1 + (P2 - pz) * n2;
            const float tt = num / dn;
            if (tt >= 0.0f) {
                const float rel0 = (px + tt * dx) - P0;
                const float rel1 = (py + tt * dy) - P1;
                const float rel2 = (pz + tt * dz) - P2;
                const float au = rel0 * J.f.eu[0] + rel1 * J.f.eu[1] + rel2 * J.f.eu[2];
                const float av = rel0 * J.f.ev[0] + rel1 * J.f.ev[1] + rel2 * J.f.ev[2];
                const float fu = au * P.idu + P.hu;
                const float fv = av * P.idv + P.hv;
                bool take = true;            // scatter filter (Section 2.4)
                if (GEN && scattered && P.scatter_filter) {
                    const uint32_t nc = n_int & 0xffffu, nr = n_int >> 16;
                    take = P.scatter_filter == 1 ? (nc == 1 && nr == 0)
                         : (P.scatter_filter == 2 ? (nr == 1 && nc == 0) : (nc + nr >= 2));
                }
                if (take && fu >= 0.0f && fu < (float)P.nu && fv >= 0.0f && fv < (float)P.nv) {
                    pixel = (int)fv * P.nu + (int)fu;
                    const long long q = llrintf(response(P, e) * 16777216.0f);
                    int64_t* t = scattered ? J.tally_s : J.tally_p;
                    atomicAdd(reinterpret_cast<unsigned long long*>(t + pixel), (unsigned long long)q);
                    outcome = scattered ? OUT_SCATTER : OUT_PRIMARY;
                }
            }
        }
        cnt.add(outcome == OUT_PRIMARY ? GDRR_ST_TALLY_PRIMARY
                                          : (outcome == OUT_SCATTER ? GDRR_ST_TALLY_SCATTER : GDRR_ST_MISS));
        record(P, outcome, pixel, 0);
        end_counts(from_inside ? 1u : 0u);
        state = S_DEAD;
    }

    __device__ __forceinline__ void move_to_box_exit(const McParams& P) {
        float te = (float)3.0e38;
        const float d[3] = {dx, dy, dz};
        const float p[3] = {px, py, pz};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (d[a] > 0.0f || d[a] < 0.0f) {
                const float t = ((d[a] > 0.0f ? P.hi[a] : P.lo[a]) - p[a]) / d[a];
                if (t < te) te = t;
            }
        }
        if (te < 0.0f) te = 0.0f;
        px = px + te * dx;
        py = py + te * dy;
        pz = pz + te * dz;
    }

    // Start flattened history g: source sampling and box entry.  Leaves the
    // lane FLY, or DEAD after tallying a photon that misses the box.
    template <class CNT>
    __device__ __forceinline__ void start(const McParams& P, uint64_t g, CNT& cnt) {
        gidx = g;
        int lo = 0, hi = P.n_jobs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (P.jobs[mid].first <= g) lo = mid; else hi = mid - 1;
        }
        job = lo;
        const Job& J = P.jobs[job];
        const uint64_t hid = J.hid_offset + (g - J.first);
        rs.init(J.angle_index, hid);
        cnt.add(GDRR_ST_HISTORIES);
        nsteps = 0;
        ngath = 0;
        scattered = 0;
        if (GEN) n_int = 0;
        if (REC) { r_virt = 0; r_ray = 0; r_comp = 0; r_first = 0; r_raymat = 0; r_dep = 0.0; }

        const uint4 w0 = rs.block(P.rk);
        const float xi_u = uniform(w0.y);
        const float xi_v = uniform(w0.z);
        const int j = cdf_search(P.kcdf_pix, P.guide_pix, P.n_guide_pix, w0.x);
        const int iu = j % P.nu, iv = j / P.nu;
        const int ecol = P.e_col ? iu : 0;   // per-column spectrum row (energy-dependent bowtie)
        const int eb = cdf_search(P.kcdf_e + ecol * P.n_bins, P.guide_e + ecol * P.n_guide_e, P.n_guide_e, w0.w);
        const float en = __ldg(P.bin_e + eb);
        if (REC) r_esrc = en;
        const float a_u = ((float)iu + xi_u - P.hu) * P.du;
        const float a_v = ((float)iv + xi_v - P.hv) * P.dv;
        const float t0 = J.f.P[0] + a_u * J.f.eu[0] + a_v * J.f.ev[0];
        const float t1 = J.f.P[1] + a_u * J.f.eu[1] + a_v * J.f.ev[1];
        const float t2 = J.f.P[2] + a_u * J.f.eu[2] + a_v * J.f.ev[2];
        dx = t0 - J.f.S[0];
        dy = t1 - J.f.S[1];
        dz = t2 - J.f.S[2];
        const float il = 1.0f / sqrtf(dx * dx + dy * dy + dz * dz);
        dx = dx * il;
        dy = dy * il;
        dz = dz * il;
        px = J.f.S[0]; py = J.f.S[1]; pz = J.f.S[2];
        e = en;

        float tmin = 0.0f, tmax = (float)3.0e38;
        bool hit = true;
        const float d[3] = {dx, dy, dz};
        const float p[3] = {px, py, pz};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (d[a] != 0.0f) {
                const float id = 1.0f / d[a];
                float t1a = (P.lo[a] - p[a]) * id;
                float t2a = (P.hi[a] - p[a]) * id;
                if (t1a > t2a) { const float t = t1a; t1a = t2a; t2a = t; }
                if (t1a > tmin) tmin = t1a;
                if (t2a < tmax) tmax = t2a;
            } else if (p[a] < P.lo[a] || p[a] > P.hi[a]) {
                hit = false;
            }
        }
        if (tmin >= tmax) hit = false;
        if (!hit) {
            escape(P, cnt, false);
            return;
        }
        px = px + tmin * dx;
        py = py + tmin * dy;
        pz = pz + tmin * dz;
        if (defer_e) need_e = true; else set_energy(P, en);
        if (LM) lm_need = LM_ALL;
        state = S_FLY;
    }

    // One Woodcock free flight and the real/virtual decision at its end.
    template <class CNT>
    __device__ __forceinline__ void step(const McParams& P, CNT& cnt) {
        if ((int)nsteps >= P.max_steps) {
            cnt.add(GDRR_ST_STEP_LIMIT);
            record(P, OUT_STEP_LIMIT, -1, 0);
            end_counts(0u);
            state = S_DEAD;
            return;
        }
        const uint4 wf = rs.block(P.rk);            // this flight's block
        const float s = -gd_logf(uniform(wf.x)) * inv_mumax;
        ++nsteps;
        if (GEN) ++c_steps;
        const float qx = px + s * dx, qy = py + s * dy, qz = pz + s * dz;
        const bool inside = (qx >= P.lo[0] && qx <= P.hi[0]) && (qy >= P.lo[1] && qy <= P.hi[1])
                         && (qz >= P.lo[2] && qz <= P.hi[2]);
        if (!inside) {
            state = S_ESC;           // the box exit and tally wait for the warp's batch
            return;
        }
        px = qx; py = qy; pz = qz;

        if (GEN && P.nearest_voxel) {
            // no density interpolation: the voxel containing the point
            const int gx = min(max((int)floorf((px - P.lo[0]) * P.ivox[0]), 0), P.nx - 1);
            const int gy = min(max((int)floorf((py - P.lo[1]) * P.ivox[1]), 0), P.ny - 1);
            const int gz = min(max((int)floorf((pz - P.lo[2]) * P.ivox[2]), 0), P.nz - 1);
            const uint2 vx = __ldg(P.vox + brick_x(gx) + brick_y(gy, P.bsy) + brick_z(gz, P.bsz));
            const float a0 = __uint_as_float(vx.x);
            const int m0 = (int)vx.y;
            const float t = uniform(wf.y) * mumax;
            if (t > a0 * cf(0, m0)) {
                ++c_virt;
                if (REC) ++r_virt;
                return;
            }
            const float muR = a0 * cf(1, m0), muC = a0 * cf(2, m0);
            m_ray = m0;
            real_collision(P, t, muR, muC, cnt);
            return;
        }

        // the lower trilinear corner, computed as gather() computes it,
        // locates the macro cell
        const int x0 = max((int)floorf((px - P.lo[0]) * P.ivox[0] - 0.5f), 0);
        const int y0 = max((int)floorf((py - P.lo[1]) * P.ivox[1] - 0.5f), 0);
        const int z0 = max((int)floorf((pz - P.lo[2]) * P.ivox[2] - 0.5f), 0);
        const float t = uniform(wf.y) * mumax;
        if (P.cells) {
            // the corners lie in [x0, x0 + 1] etc., inside the cover of x0's cell:
            // above the cell's bound the collision is virtual whatever they hold
            const int cell = (x0 >> P.cshift) + P.csx * ((y0 >> P.cshift) + P.csy * (z0 >> P.cshift));
            if (t > cell_bound(P, cell)) {
                if (GEN) { ++c_virt; ++c_skip; }
                if (REC) ++r_virt;
                return;
            }
        }
        // the corner gathers wait for the warp's service batch
        tg = t;
        if (GEN) wz = wf.z;
        state = S_GATHER;
    }

    // The boundary plane between cells j - 1 and j of axis a (n cells): the
    // box faces for j = 0 and j = n, else where the lower trilinear corner
    // index reaches j 2^s, i.e. (x - lo) / vox - 1/2 = j 2^s.
    __device__ __forceinline__ static float lm_plane(const McParams& P, int a, int j, int n) {
        if (j <= 0) return P.lo[a];
        if (j >= n) return P.hi[a];
        return P.lo[a] + ((float)(j << P.cshift) + 0.5f) * P.vox_mm[a];
    }

    // LM, in the service batch: the entry cell of a new history, the
    // reciprocals of a new direction, and the next flight: its Philox block,
    // its optical depth tau = -ln xi and the uniform of its ordinate test.
    template <class CNT>
    __device__ __forceinline__ void lm_prepare(const McParams& P, CNT& cnt) {
        if (lm_need & LM_CELL) {
            const int gx = max((int)floorf((px - P.lo[0]) * P.ivox[0] - 0.5f), 0) >> P.cshift;
            const int gy = max((int)floorf((py - P.lo[1]) * P.ivox[1] - 0.5f), 0) >> P.cshift;
            const int gz = max((int)floorf((pz - P.lo[2]) * P.ivox[2] - 0.5f), 0) >> P.cshift;
            cx = min(gx, P.ncx - 1);
            cy = min(gy, P.ncy - 1);
            cz = min(gz, P.ncz - 1);
        }
        if (lm_need & LM_DIR) {
            idx = dx != 0.0f ? 1.0f / dx : 0.0f;
            idy = dy != 0.0f ? 1.0f / dy : 0.0f;
            idz = dz != 0.0f ? 1.0f / dz : 0.0f;
        }
        lm_need = 0u;
        if ((int)nsteps >= P.max_steps) {
            cnt.add(GDRR_ST_STEP_LIMIT);
            record(P, OUT_STEP_LIMIT, -1, 0);
            end_counts(0u);
            state = S_DEAD;
            return;
        }
        const uint4 wf = rs.block(P.rk);
        ++nsteps;
        if (GEN) ++c_steps;
        tau = -log_uniform((wf.x >> 8) + 1u);
        tg = uniform(wf.y);
        if (GEN) wz = wf.z;
    }

    // LM: one cell of a flight.  With b the cell's bound and tx the distance
    // to its exit, the remaining depth either runs out inside (the tentative
    // collision lies tau / b ahead and waits for the warp's service batch) or
    // pays b tx, and the lane moves to the exit point and on to the next cell
    // (one step along every axis whose exit plane is nearest, all of them on
    // a tie).  Every crossing moves the cell along the direction of flight, so
    // a flight crosses at most ncx + ncy + ncz cells; leaving the grid leaves
    // the box, from the last position inside.
    __device__ __forceinline__ void walk(const McParams& P, float b) {
        // distance to the cell's exit plane of an axis (0 when already on it)
        auto exit_at = [&](int ax, int c, int n, float d, float p, float id) {
            const float l = (lm_plane(P, ax, d > 0.0f ? c + 1 : c, n) - p) * id;
            return d != 0.0f ? (l > 0.0f ? l : 0.0f) : (float)3.0e38;
        };
        const float tx = exit_at(0, cx, P.ncx, dx, px, idx), ty = exit_at(1, cy, P.ncy, dy, py, idy),
                    tz = exit_at(2, cz, P.ncz, dz, pz, idz);
        const float t = fminf(tx, fminf(ty, tz));
        const float bt = b * t;
        if (tau < bt) {
            const float s = tau / b;
            px = px + s * dx;
            py = py + s * dy;
            pz = pz + s * dz;
            tg = tg * b;
            state = S_GATHER;
            return;
        }
        tau = tau - bt;
        const bool sx = dx != 0.0f && tx == t, sy = dy != 0.0f && ty == t, sz = dz != 0.0f && tz == t;
        const int nx_ = sx ? cx + (dx > 0.0f ? 1 : -1) : cx;
        const int ny_ = sy ? cy + (dy > 0.0f ? 1 : -1) : cy;
        const int nz_ = sz ? cz + (dz > 0.0f ? 1 : -1) : cz;
        if (!(sx || sy || sz) || nx_ < 0 || nx_ >= P.ncx || ny_ < 0 || ny_ >= P.ncy || nz_ < 0 || nz_ >= P.ncz) {
            state = S_ESC;
            return;
        }
        px = px + t * dx;
        py = py + t * dy;
        pz = pz + t * dz;
        cx = nx_; cy = ny_; cz = nz_;
        ++c_cross;
    }

    // The deferred part of a free flight that passed the macro-cell test:
    // the eight-corner mixture at the lane's position and the real/virtual
    // decision for its t.  The warp serves its waiting lanes together, so the
    // gathers run on many lanes at once instead of on the few whose flights
    // passed the test in one iteration.
    template <class CNT>
    __device__ __forceinline__ void gather(const McParams& P, CNT& cnt) {
        if (!GEN) ++ngath;
        const float t = tg;
        if (GEN && P.nearest_voxel) {
            // no density interpolation: the voxel containing the point
            const int gx = min(max((int)floorf((px - P.lo[0]) * P.ivox[0]), 0), P.nx - 1);
            const int gy = min(max((int)floorf((py - P.lo[1]) * P.ivox[1]), 0), P.ny - 1);
            const int gz = min(max((int)floorf((pz - P.lo[2]) * P.ivox[2]), 0), P.nz - 1);
            const uint2 vx = __ldg(P.vox + brick_x(gx) + brick_y(gy, P.bsy) + brick_z(gz, P.bsz));
            const float a0 = __uint_as_float(vx.x);
            const int m0 = (int)vx.y;
            if (t > a0 * total(m0)) {
                ++c_virt;
                if (REC) ++r_virt;
                lm_need |= LM_DRAW;
                state = S_FLY;
                return;
            }
            m_ray = m0;
            real_collision(P, t, a0 * cf(1, m0), a0 * cf(2, m0), cnt);
            return;
        }
        float a[8];
        int mc[8];
        corners(P, px, py, pz, a, mc);
        float muT = a[0] * total(mc[0]);
#pragma unroll
        for (int c = 1; c < 8; ++c) muT = muT + a[c] * total(mc[c]);
        if (t > muT) {
            ++c_virt;
            if (REC) ++r_virt;
            if (LM) lm_need |= LM_DRAW;
            state = S_FLY;
            return;
        }
        float muR = a[0] * cf(1, mc[0]);
#pragma unroll
        for (int c = 1; c < 8; ++c) muR = muR + a[c] * cf(1, mc[c]);
        float muC = a[0] * cf(2, mc[0]);
#pragma unroll
        for (int c = 1; c < 8; ++c) muC = muC + a[c] * cf(2, mc[c]);
        if (GEN && P.ray_ff && t <= muR) {
            // the form factor's material: the corner whose Rayleigh share of
            // mu_R holds xi mu_R, xi the flight block's third word
            const float target = uniform(wz) * muR;
            float acc = 0.0f;
            m_ray = mc[7];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                acc = acc + a[c] * cf(1, mc[c]);
                if (target <= acc) { m_ray = mc[c]; break; }
            }
        }
        real_collision(P, t, muR, muC, cnt);
    }

    // A real collision: Rayleigh if t <= mu_R, Compton if t <= mu_R + mu_C,
    // else photoelectric absorption.
    template <class CNT>
    __device__ __forceinline__ void real_collision(const McParams& P, float t, float muR, float muC, CNT& cnt) {
        if (t <= muR) {
            state = S_RAY;
        } else if (t <= muR + muC) {
            state = S_COMP;
        } else {
            cnt.add(GDRR_ST_PHOTO);
            if (REC) { if (!r_first) r_first = 3; r_dep += (double)e; }
            record(P, OUT_PHOTO, -1, 1);
            end_counts(0u);
            state = S_DEAD;
        }
    }

    // The deferred Rayleigh or Compton interaction of a waiting lane.  The
    // polar angle comes from the event's own sampler; the azimuth and the
    // rotation are common code, so a batch holding both kinds runs them once.
    template <class CNT>
    __device__ __forceinline__ void interact(const McParams& P, CNT& cnt) {
        const bool ray = state == S_RAY;
        float ct, e2 = e;
        if (GEN && ray && P.ray_ff) {
            ct = rayleigh_ff(rs, P, e, m_ray);
            if (REC) r_raymat = (uint32_t)m_ray;
        } else {
            polar(rs, P.rk, ray, e, ct, e2);
        }
        float cp, sp;
        azimuth(rs, P.rk, cp, sp);
        rotate(dx, dy, dz, ct, cp, sp);
        scattered = 1;
        if (ray) {
            if (GEN) n_int += 0x10000u;
            cnt.add(GDRR_ST_RAYLEIGH);
            if (REC) { ++r_ray; if (!r_first) r_first = 1; }
            if (LM) lm_need |= LM_DRAW | LM_DIR;
            state = S_FLY;
            return;
        }
        if (GEN) n_int += 1u;
        cnt.add(GDRR_ST_COMPTON);
        if (REC) { ++r_comp; if (!r_first) r_first = 2; r_dep += (double)e - (double)e2; }
        if (e2 < P.e_cut) {
            e = e2;
            if (REC) r_dep += (double)e;
            cnt.add(GDRR_ST_CUTOFF);
            record(P, OUT_CUTOFF, -1, 0);
            end_counts(0u);
            state = S_DEAD;
            return;
        }
        if (defer_e) {
            e = e2;
            need_e = true;
        } else {
            set_energy(P, e2);
        }
        if (LM) lm_need |= LM_DRAW | LM_DIR;
        state = S_FLY;
    }
};

// The transport with records (parity runs): one photon per lane from birth to
// death.
template <int NM, bool GEN, bool LM>
// Up to 512 threads per block, 64 registers per thread (the same cap at 2 x 512
// or 4 x 256 resident threads): the autotuner's block sizes 64 ... 512.
__global__ void __launch_bounds__(512, 2) mc_kernel(const McParams P) {
    extern __shared__ float smem[];
    __shared__ unsigned long long counts[GDRR_NSTATS];
    for (int i = threadIdx.x; i < GDRR_NSTATS; i += blockDim.x) counts[i] = 0ull;
    __syncthreads();

    const int lane = threadIdx.x & 31;
    SharedCounts cnt = {counts};
    Lane<NM, true, GEN, LM> L;
    L.coef = smem + threadIdx.x;
    L.stride = blockDim.x;
    L.tot = L.coef;
    L.tot_stride = L.stride;
    L.state = S_DEAD;
    L.defer_e = true;                 // new histories and Compton events share one table pass
    L.need_e = false;
    L.c_steps = 0; L.c_virt = 0; L.c_skip = 0;
    L.lm_need = 0u; L.c_cross = 0u;
    unsigned long long pool_next = 0, pool_end = 0;
    bool exhausted = false;

    for (;;) {
        const unsigned fly = __ballot_sync(FULL, L.state == S_FLY);
        if (32 - __popc(fly) >= P.batch_min || fly == 0u) {
            // serve waiting lanes together: corner gathers, interactions,
            // tallies, new histories
            if (L.state == S_GATHER) L.gather(P, cnt);
            if (L.state == S_RAY || L.state == S_COMP) L.interact(P, cnt);
            if (L.state == S_ESC) L.escape(P, cnt, true);
            if (!exhausted) {
                unsigned need = __ballot_sync(FULL, L.state == S_DEAD);
                while (need) {
                    if (pool_next >= pool_end) {
                        unsigned long long base = 0;
                        if (lane == 0) base = atomicAdd(P.counter, (unsigned long long)P.chunk);
                        base = __shfl_sync(FULL, base, 0);
                        if (base >= P.total) { exhausted = true; break; }
                        pool_next = base;
                        pool_end = base + (unsigned long long)P.chunk;
                        if (pool_end > P.total) pool_end = P.total;
                    }
                    const unsigned avail = (unsigned)(pool_end - pool_next);
                    const unsigned want = (unsigned)__popc(need);
                    const unsigned take = want < avail ? want : avail;
                    const unsigned rank = (unsigned)__popc(need & ((1u << lane) - 1u));
                    if (((need >> lane) & 1u) && rank < take) L.start(P, pool_next + rank, cnt);
                    pool_next += take;
                    need = __ballot_sync(FULL, L.state == S_DEAD);
                }
            }
            if (L.need_e) {
                L.set_energy(P, L.e);
                L.need_e = false;
            }
            if (LM && L.lm_need) L.lm_prepare(P, cnt);
            if (exhausted && !__any_sync(FULL, L.state != S_DEAD)) break;
        }
        if (L.state == S_FLY) {
            if constexpr (LM) L.walk(P, L.cell_bound(P, L.cx + P.csx * (L.cy + P.csy * L.cz)));
            else L.step(P, cnt);
        }
    }

    atomicAdd(&counts[GDRR_ST_STEPS], (unsigned long long)L.c_steps);
    atomicAdd(&counts[GDRR_ST_VIRTUAL], (unsigned long long)L.c_virt);
    atomicAdd(&counts[GDRR_ST_CELL_SKIPS], (unsigned long long)L.c_skip);
    if (LM) atomicAdd(&counts[GDRR_ST_CELL_CROSSINGS], (unsigned long long)L.c_cross);
    __syncthreads();
    for (int i = threadIdx.x; i < GDRR_NSTATS; i += blockDim.x)
        if (counts[i]) atomicAdd(P.stats + i, counts[i]);
}

// ---------------------------------------------------------------------------
// The transport without records: a pool of photons per warp.
//
// A lane that keeps its photon from birth to death (mc_kernel) waits while
// its warp serves others and serves its rare events on partial warps: 16 of
// 32 lanes were active per instruction.  Here a warp owns a pool of photons
// (more than its 32 lanes) in shared memory and four lists of them: ready to
// fly, at a tentative collision (the corner gathers), at a real one (the
// interaction), and at the end of their history (the box exit and tally, then
// the next history).  It flies 32 photons at a time; a lane whose flight stops
// hands its photon to a list and takes the next ready one, and once a list
// holds a whole warp's worth, the warp parks its photons and serves that list
// with every lane.  Nothing is shared between warps, so there is no block
// barrier: lists and slots are exchanged under __syncwarp alone.
//
// The arithmetic per photon is Lane's (start, gather, interact, escape, walk)
// or, for the free flight, the same operations on fewer instructions, so every
// history's draws, decisions and tally are the ones mc_kernel and the oracle
// produce; integer tallies and counters do not depend on the order in which
// histories advance.
//
// The flight loop loads the macro-cell record of its end point first and forms
// the next flight's Philox block and logarithm while the load is under way; a
// photon carries those words through its slot, and only a collision or a new
// history, whose blocks move on, forms them anew.
//
// What bounds it: instruction issue (67 to 71 % of the slots, 25 of 32 lanes active
// per instruction, 28 in flight) beside L1 wavefronts (63 %).  2 mm torso, 1e8
// histories (46 free flights each): 75.3 ms with one photon per lane and a
// separate source pass, 50.3 ms so; per history 725 warp instructions before and
// 470 now.  Of a warp's time 40 % are free flights, 12 % hand-overs, 12 % gathers,
// 15 % interactions and 10 % tallies and starts.
//
// A slot is Q float4 words: {px py pz, and t = xi mumax at a tentative
// collision or the next flight's -ln xi} {dx dy dz E} {mumax 1/mumax, or the
// optical depth and cell x of LM; history id lo; job, flags} {blocks drawn,
// block limit, history id hi, the next flight's second word or LM's cell y}
// {total coefficient per material}, LM {1/d, cell z}, GEN {the flight's third word,
// interaction counts, form-factor material}.  The history's free flights so
// far are its blocks less those drawn elsewhere, so the flight only compares
// its block number with a limit that grows by the blocks drawn elsewhere:
// max_steps costs no counter of its own.  The totals of free flights, and of
// the virtual collisions the cells decided, follow from warp-wide counts of
// lanes per iteration.
constexpr int WARP_BLOCK = 32 * POOL_WARPS;   // threads; the warps of a block share nothing but counters
// Idle lanes at which the warp hands over and refills: 5, 6, 8 and 12 were
// within 2 %, 4 was 3 % slower (a hand-over costs about half a flight).
constexpr int REFILL_IDLE = 8;
// With local majorants a third of the flights stop in every cell, so a refill at 8
// would come after each: 2e7 histories of the 2 mm torso take 12.9 ms at 8, 12.7 at
// 14, 12.5 at 18, 12.4 from 20 to 24, 12.6 at 26 and 13.5 at 30.
constexpr int REFILL_IDLE_LM = 22;
// a slot's flags beside its job
constexpr uint32_t JF_SCATTERED = 0x80000000u, JF_DEAD = 0x40000000u, JF_RAYLEIGH = 0x20000000u, JF_JOB = 0x1fffffffu;

template <int NM, bool GEN, bool LM>
struct Slots {
    static constexpr int CF = NM < 4 ? 1 : NM / 4;              // float4 words of the total coefficients
    static constexpr int Q_LM = 4 + CF, Q_GEN = Q_LM + (LM ? 1 : 0), Q = Q_GEN + (GEN ? 1 : 0);
    static_assert(Q == slot_words(NM, GEN, LM), "the rules' size of a slot");
    float4* s;
    __device__ __forceinline__ float4& at(int slot, int q) const { return s[slot * Q + q]; }
    __device__ __forceinline__ uint32_t& word(int slot, int q, int w) const {
        return reinterpret_cast<uint32_t*>(s)[(slot * Q + q) * 4 + w];
    }
    __device__ __forceinline__ void totals(int slot, float (&t)[NM]) const {
        if constexpr (NM == 2) {
            const float4 v = at(slot, 4);
            t[0] = v.x; t[1] = v.y;
        } else {
#pragma unroll
            for (int q = 0; q < CF; ++q) {
                const float4 v = at(slot, 4 + q);
                t[4 * q] = v.x; t[4 * q + 1] = v.y; t[4 * q + 2] = v.z; t[4 * q + 3] = v.w;
            }
        }
    }
    __device__ __forceinline__ void set_totals(int slot, const float (&t)[NM]) const {
        if constexpr (NM == 2) {
            at(slot, 4) = make_float4(t[0], t[1], 0.0f, 0.0f);
        } else {
#pragma unroll
            for (int q = 0; q < CF; ++q) at(slot, 4 + q) = make_float4(t[4 * q], t[4 * q + 1], t[4 * q + 2], t[4 * q + 3]);
        }
    }
};

// a lane's photon: none, in flight, at a tentative collision, out of the box,
// at max_steps
enum : int { F_NONE = 0, F_ON = 1, F_GATHER = 2, F_ESC = 3, F_LIMIT = 4 };
// a warp's counts: the statistics, then the flights that stopped at a
// tentative collision and outside the box
enum : int { A_GATHER = GDRR_NSTATS, A_ESC, A_N };
static_assert(A_N == POOL_COUNTS, "the rules' size of a warp's counts");

// One row of the energy-major coefficient table [energy][kind][NM].
template <int NM>
__device__ __forceinline__ void coef_row(const float* __restrict__ t, float (&v)[NM]) {
    if constexpr (NM == 2) {
        const float2 a = __ldg(reinterpret_cast<const float2*>(t));
        v[0] = a.x; v[1] = a.y;
    } else {
#pragma unroll
        for (int q = 0; q < NM; q += 4) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(t + q));
            v[q] = a.x; v[q + 1] = a.y; v[q + 2] = a.z; v[q + 3] = a.w;
        }
    }
}

// The coefficients of kind k (0 Rayleigh, 1 Compton, 2 photoelectric) of every
// material at energy node ie plus fraction f, as Lane::set_energy takes them.
template <int NM>
__device__ __forceinline__ void coef_kind(const McParams& P, int k, int ie, float f, float (&v)[NM]) {
    float a[NM], b[NM];
    coef_row<NM>(P.tab_e + (size_t)(ie * 3 + k) * NM, a);
    coef_row<NM>(P.tab_e + (size_t)(ie * 3 + 3 + k) * NM, b);
#pragma unroll
    for (int m = 0; m < NM; ++m) v[m] = a[m] + f * (b[m] - a[m]);
}

// Lane::set_energy's totals and majorant, without its shared-memory table.
template <int NM>
__device__ __forceinline__ void energy_totals(const McParams& P, float e, float (&t)[NM], float& mumax) {
    int ie; float f;
    interp_index(e, P.e0, P.inv_de, P.n_e, ie, f);
    float c[NM], p[NM];
    coef_kind<NM>(P, 0, ie, f, t);
    coef_kind<NM>(P, 1, ie, f, c);
    coef_kind<NM>(P, 2, ie, f, p);
#pragma unroll
    for (int m = 0; m < NM; ++m) t[m] = (t[m] + c[m]) + p[m];
    const float a = __ldg(P.major + ie), b = __ldg(P.major + ie + 1);
    mumax = a > b ? a : b;
}

// A flight's Philox block on 35 of the 40 operations of philox4x32_10: only
// the block number changes along a history, so the part of the first two
// rounds that it does not reach is formed once per hand-over (flight_keys),
// and the last round's words z, w are dropped where unused.
struct FlightKeys { uint32_t a, b, c, d; };

__device__ __forceinline__ FlightKeys flight_keys(uint32_t angle, uint32_t hlo, uint32_t hhi, const RoundKeys& rk) {
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * hlo;
    const uint64_t p0 = (uint64_t)0xD2511F53u * ((uint32_t)(p1 >> 32) ^ angle ^ rk.k0[0]);
    FlightKeys k;
    k.a = hhi ^ rk.k1[0];
    k.b = (uint32_t)p1 ^ rk.k0[1];
    k.c = (uint32_t)(p0 >> 32) ^ rk.k1[1];
    k.d = (uint32_t)p0;
    return k;
}

__device__ __forceinline__ uint4 flight_block(uint32_t blk, const FlightKeys& k, const RoundKeys& rk) {
    const uint64_t q0 = (uint64_t)0xD2511F53u * blk;
    const uint64_t q1 = (uint64_t)0xCD9E8D57u * ((uint32_t)(q0 >> 32) ^ k.a);
    uint32_t c0 = (uint32_t)(q1 >> 32) ^ k.b, c1 = (uint32_t)q1, c2 = k.c ^ (uint32_t)q0, c3 = k.d;
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ rk.k0[r];
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ rk.k1[r];
        c0 = n0; c1 = (uint32_t)p1; c2 = n2; c3 = (uint32_t)p0;
    }
    return make_uint4(c0, c1, c2, c3);
}

// 0x4b000000 + floor(y - 1/2) for y = (x - lo) / vox >= 0: adding 2^23 - 1/2
// with rounding down leaves the floor in the low bits (the sum is formed
// exactly before it is rounded, and floorf(y - 0.5f) is the same floor: y -
// 1/2 is exact for y >= 1/2, and lies in [-1/2, 0) below).  The lower corner
// -1 of a point in the outer half voxel needs no clamp: its cell, -1, is a
// copy of cell 0 in the table.
__device__ __forceinline__ uint32_t corner_bits(float y) { return __float_as_uint(__fadd_rd(y, 8388607.5f)); }

// The macro cell of a point inside the box: that of its lower trilinear corner,
// as gather() computes it (cell0: the number that corner_bits' offset makes of
// cell 0).
__device__ __forceinline__ int cell_at(const McParams& P, float x, float y, float z, uint32_t cell0) {
    const uint32_t ux = corner_bits((x - P.lo[0]) * P.ivox[0]) >> P.cshift;
    const uint32_t uy = corner_bits((y - P.lo[1]) * P.ivox[1]) >> P.cshift;
    const uint32_t uz = corner_bits((z - P.lo[2]) * P.ivox[2]) >> P.cshift;
    return (int)(ux + P.csx * (uy + P.csy * uz) - cell0);
}

// The macro-cell bound (Lane::cell_bound) from the cell's densities.
template <int NM>
__device__ __forceinline__ float bound_of(const float (&v)[NM], const float (&cf)[NM]) {
    float b = v[0] * cf[0];
#pragma unroll
    for (int m = 1; m < NM; ++m) b = fmaxf(b, v[m] * cf[m]);
    return b * CELL_MARGIN;
}

template <int NM>
__device__ __forceinline__ float bound_of(const McParams& P, int cell, const float (&cf)[NM]) {
    float v[NM];
    coef_row<NM>(P.cells + (ptrdiff_t)cell * NM, v);
    return bound_of<NM>(v, cf);
}



template <int NM, bool GEN, bool LM>
__global__ void __launch_bounds__(WARP_BLOCK, pool_blocks(NM, GEN, LM)) mc_warp_kernel(
    const McParams P, int n_pool, int n_use, unsigned chunk, uint32_t cell0) {
    extern __shared__ __align__(16) unsigned char warp_smem[];
    __shared__ unsigned long long cnt[GDRR_NSTATS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    for (int i = threadIdx.x; i < GDRR_NSTATS; i += WARP_BLOCK) cnt[i] = 0ull;
    __syncthreads();
    unsigned char* base = warp_smem + (size_t)warp * pool_bytes(n_pool, NM, GEN, LM);
    Slots<NM, GEN, LM> S;
    S.s = reinterpret_cast<float4*>(base);
    float* coef = reinterpret_cast<float*>(base + (size_t)n_pool * S.Q * 16) + lane;       // [2 NM][32], this lane's column
    uint8_t* qR = base + (size_t)n_pool * S.Q * 16 + (size_t)2 * NM * 32 * 4;               // ready to fly
    uint8_t* qG = qR + n_pool;                                                             // corner gathers
    uint8_t* qI = qG + n_pool;                                                             // interaction
    uint8_t* qE = qI + n_pool;                                                             // tally and next history
    int nR = 0, nG = 0, nI = 0, nE = n_use;
    for (int i = lane; i < n_use; i += 32) {
        qE[i] = (uint8_t)i;
        S.word(i, 2, 3) = JF_DEAD;
    }
    __syncwarp();
    // this warp's counts of events, by kind; histories claimed and not started
    unsigned long long* acc = reinterpret_cast<unsigned long long*>(qR + 4 * n_pool);
    unsigned long long &next = acc[A_N], &end = acc[A_N + 1];
    if (lane < A_N + 2) acc[lane] = 0ull;
    __syncwarp();
    bool exhausted = false;
    auto add = [&](int k, unsigned n) {
        if (lane == 0) acc[k] += n;
    };
    auto tally = [&](int k, bool p) { add(k, (unsigned)__popc(__ballot_sync(FULL, p))); };
    Lane<NM, false, GEN, LM> L;
    L.coef = coef - NM * 32;                // kinds 1 and 2; the totals are the slot's
    L.stride = 32;
    L.tot_stride = 1;
    L.defer_e = true;
    L.c_steps = 0; L.c_virt = 0; L.c_skip = 0; L.c_cross = 0; L.ngath = 0; L.lm_need = 0u;

    for (;;) {
        const int most = max(max(nG, nI), nE);
        if (most < 32 && (most == 0 || most < nR)) {
            if (nR == 0) break;
            // ---- free flights: until a list is full, or too few photons fly ----
            float cf[NM];
            float mumax = 0.0f, inv = 0.0f, nl = 0.0f;     // nl, wy, wz: the next flight's -ln xi and words
            uint32_t blk = 0, limit = 0, wy = 0, wz = 0, gz = 0;
            FlightKeys key = {0, 0, 0, 0};
            int slot = 0, code = F_NONE;
            unsigned flown = 0, crossed = 0, drawn = 0, celled = 0;
            for (;;) {
                const unsigned act = __ballot_sync(FULL, code == F_ON);
                int n_act = __popc(act);
                if (n_act <= 32 - (LM ? REFILL_IDLE_LM : REFILL_IDLE)) {
                    // hand over the photons whose flight stopped, refill the lanes
                    const unsigned mG = __ballot_sync(FULL, code == F_GATHER), mE = __ballot_sync(FULL, code >= F_ESC);
                    if (code > F_ON) {
                        S.at(slot, 0) = make_float4(L.px, L.py, L.pz, L.tg);
                        if constexpr (LM) {
                            S.word(slot, 2, 1) = (uint32_t)L.cx;
                            S.word(slot, 3, 3) = (uint32_t)L.cy;
                            S.word(slot, S.Q_LM, 3) = (uint32_t)L.cz;
                        } else {
                            S.word(slot, 3, 0) = blk;
                            if (GEN) S.word(slot, S.Q_GEN, 0) = gz;
                            if (code == F_LIMIT) S.word(slot, 2, 3) = JF_DEAD;
                        }
                        if (code == F_GATHER) qG[nG + __popc(mG & below)] = (uint8_t)slot;
                        else qE[nE + __popc(mE & below)] = (uint8_t)slot;
                    }
                    nG += __popc(mG);
                    nE += __popc(mE);
                    const unsigned cut = LM ? 0u : __ballot_sync(FULL, code == F_LIMIT);
                    if (cut) {
                        add(GDRR_ST_STEP_LIMIT, (unsigned)__popc(cut));
                        flown -= (unsigned)__popc(cut);
                    }
                    if (code > F_ON) code = F_NONE;
                    const int full = max(max(nG, nI), nE);
                    if (full >= 32 || (nR == 0 && n_act <= full)) break;
                    __syncwarp();
                    const int take = nR - 1 - __popc(~act & below);
                    if (code == F_NONE && take >= 0) {
                        code = F_ON;
                        slot = qR[take];
                        const float4 a = S.at(slot, 0), b = S.at(slot, 1), c = S.at(slot, 2);
                        L.px = a.x; L.py = a.y; L.pz = a.z;
                        L.dx = b.x; L.dy = b.y; L.dz = b.z;
                        S.totals(slot, cf);
                        if constexpr (LM) {
                            const float4 g = S.at(slot, S.Q_LM);
                            L.tg = a.w;
                            L.tau = c.x;
                            L.cx = __float_as_int(c.y);
                            L.cy = (int)S.word(slot, 3, 3);
                            L.idx = g.x; L.idy = g.y; L.idz = g.z;
                            L.cz = __float_as_int(g.w);
                        } else {
                            const float4 d = S.at(slot, 3);
                            nl = a.w;
                            mumax = c.x; inv = c.y;
                            blk = __float_as_uint(d.x); limit = __float_as_uint(d.y); wy = __float_as_uint(d.w);
                            if (GEN) wz = S.word(slot, S.Q_GEN, 0);
                            key = flight_keys(P.jobs[__float_as_uint(c.w) & JF_JOB].angle_index, __float_as_uint(c.z),
                                              __float_as_uint(d.z), P.rk);
                        }
                    }
                    n_act = min(32, n_act + nR);
                    nR = max(0, nR - __popc(~act));
                }
                flown += (unsigned)n_act;
                bool again = false, over = false;
                if (code == F_ON) {
                    if constexpr (LM) {
                        L.state = S_FLY;
                        L.walk(P, bound_of<NM>(P, L.cx + P.csx * (L.cy + P.csy * L.cz), cf));
                        code = L.state == S_FLY ? F_ON : (L.state == S_GATHER ? F_GATHER : F_ESC);
                        if (GEN && P.in_place && code == F_GATHER && !P.nearest_voxel) {
                            // coarse cells: the mixture and a virtual collision's next
                            // flight here (a history at max_steps ends in the service)
                            float a[8];
                            int mc[8];
                            corners(P, L.px, L.py, L.pz, a, mc);
                            float mu = a[0] * __uint_as_float(S.word(slot, 4, mc[0]));
#pragma unroll
                            for (int c = 1; c < 8; ++c) mu = mu + a[c] * __uint_as_float(S.word(slot, 4, mc[c]));
                            const uint32_t b = S.word(slot, 3, 0);
                            if (L.tg > mu && b < S.word(slot, 3, 1)) {
                                const uint4 w = flight_block(
                                    b, flight_keys(P.jobs[S.word(slot, 2, 3) & JF_JOB].angle_index, S.word(slot, 2, 2),
                                                   S.word(slot, 3, 2), P.rk), P.rk);
                                S.word(slot, 3, 0) = b + 1u;
                                S.word(slot, S.Q_GEN, 0) = w.z;
                                L.tau = -log_uniform((w.x >> 8) + 1u);
                                L.tg = uniform(w.y);
                                code = F_ON;
                                again = true;
                            }
                        }
                    } else {
                        const float s = nl * inv;
                        const float qx = L.px + s * L.dx, qy = L.py + s * L.dy, qz = L.pz + s * L.dz;
                        const bool inside = fabsf(qx) <= P.hi[0] && fabsf(qy) <= P.hi[1] && fabsf(qz) <= P.hi[2];  // lo = -hi
                        const float t = uniform(wy) * mumax;
                        // what decides a tentative collision is loaded first ...
                        float v[NM];
                        uint2 vx = make_uint2(0u, 0u);
                        const bool nearest = GEN && P.nearest_voxel, here = GEN && P.in_place;
                        float mu = 0.0f;
                        if (here && !nearest) {
                            // no cells, or cells so coarse that few collisions are virtual by their
                            // bound: the mixture itself, here where nearly all are virtual, and the
                            // bound (never below it) for the count of those it decides
                            if (inside) {
                                float a[8];
                                int mc[8];
                                corners(P, qx, qy, qz, a, mc);
                                mu = a[0] * __uint_as_float(S.word(slot, 4, mc[0]));
#pragma unroll
                                for (int c = 1; c < 8; ++c) mu = mu + a[c] * __uint_as_float(S.word(slot, 4, mc[c]));
                                if (P.cells != P.open_cell)
                                    over = t > bound_of<NM>(P, cell_at(P, qx, qy, qz, cell0), cf);
                            }
                        } else if (nearest) {
                            const int gx = min(max((int)floorf((qx - P.lo[0]) * P.ivox[0]), 0), P.nx - 1);
                            const int gy = min(max((int)floorf((qy - P.lo[1]) * P.ivox[1]), 0), P.ny - 1);
                            const int gv = min(max((int)floorf((qz - P.lo[2]) * P.ivox[2]), 0), P.nz - 1);
                            vx = __ldg(P.vox + brick_x(gx) + brick_y(gy, P.bsy) + brick_z(gv, P.bsz));
                        } else {
                            const int cell = cell_at(P, qx, qy, qz, cell0);
                            coef_row<NM>(P.cells + (ptrdiff_t)(inside ? cell : 0) * NM, v);
                        }
                        // ... and the next flight's words formed while it comes
                        const bool cut = blk >= limit;
                        ++blk;
                        if (GEN) gz = wz;
                        const uint4 w = flight_block(blk, key, P.rk);
                        nl = -log_uniform((w.x >> 8) + 1u);
                        wy = w.y;
                        if (GEN) wz = w.z;
                        const bool skip = t > (nearest ? __uint_as_float(vx.x) * __uint_as_float(S.word(slot, 4, (int)vx.y))
                                                       : here ? mu : bound_of<NM>(v, cf));
                        L.tg = t;
                        if (inside) { L.px = qx; L.py = qy; L.pz = qz; }
                        code = skip ? F_ON : F_GATHER;
                        if (!inside) code = F_ESC;
                        if (cut) code = F_LIMIT;
                    }
                }
                if (LM) crossed += (unsigned)__popc(__ballot_sync(FULL, code == F_ON && !again));
                if (LM && GEN) drawn += (unsigned)__popc(__ballot_sync(FULL, again));
                if (!LM && GEN && P.in_place) celled += (unsigned)__popc(__ballot_sync(FULL, code == F_ON && over));
            }
            // park the photons still in flight
            __syncwarp();
            const unsigned fly = __ballot_sync(FULL, code == F_ON);
            if (code == F_ON) {
                S.at(slot, 0) = make_float4(L.px, L.py, L.pz, LM ? L.tg : nl);
                if constexpr (LM) {
                    S.word(slot, 2, 0) = __float_as_uint(L.tau);
                    S.word(slot, 2, 1) = (uint32_t)L.cx;
                    S.word(slot, 3, 3) = (uint32_t)L.cy;
                    S.word(slot, S.Q_LM, 3) = (uint32_t)L.cz;
                } else {
                    S.word(slot, 3, 0) = blk;
                    S.word(slot, 3, 3) = wy;
                    if (GEN) S.word(slot, S.Q_GEN, 0) = wz;
                }
                qR[nR + __popc(fly & below)] = (uint8_t)slot;
            }
            nR += __popc(fly);
            add(LM ? GDRR_ST_CELL_CROSSINGS : GDRR_ST_STEPS, LM ? crossed : flown);
            if (!LM && GEN) add(GDRR_ST_CELL_SKIPS, celled);
            if (LM && GEN) {
                add(GDRR_ST_STEPS, drawn);
                add(GDRR_ST_VIRTUAL, drawn);
            }
            __syncwarp();
            continue;
        }

        // ---- services: the fullest list's last 32, or what there is ------------
        const int which = nI >= nG && nI >= nE ? S_COMP : (nG >= nE ? S_GATHER : S_ESC);
        const int have = which == S_COMP ? nI : (which == S_GATHER ? nG : nE), n = min(32, have);
        int slot = -1;
        if (lane < n) slot = (which == S_COMP ? qI : (which == S_GATHER ? qG : qE))[have - 1 - lane];
        if (which == S_COMP) nI -= n; else if (which == S_GATHER) nG -= n; else nE -= n;
        __syncwarp();
        EventMask ev = {0u};
        bool fresh = false;                       // a new energy: totals and majorant to form
        float4 c = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        uint32_t limit = 0, jf = JF_DEAD;
        L.state = S_DEAD;
        if (slot >= 0) {
            c = S.at(slot, 2);
            jf = __float_as_uint(c.w);
            if (!(jf & JF_DEAD)) {
                const float4 a = S.at(slot, 0), b = S.at(slot, 1), d = S.at(slot, 3);
                L.px = a.x; L.py = a.y; L.pz = a.z; L.tg = a.w;
                L.dx = b.x; L.dy = b.y; L.dz = b.z; L.e = b.w;
                L.job = (int)(jf & JF_JOB);
                L.scattered = (jf & JF_SCATTERED) ? 1 : 0;
                L.rs.angle = P.jobs[L.job].angle_index;
                L.rs.hlo = __float_as_uint(c.z);
                L.rs.hhi = __float_as_uint(d.z);
                L.rs.blk = __float_as_uint(d.x);
                limit = __float_as_uint(d.y);
                if (GEN) {
                    L.wz = S.word(slot, S.Q_GEN, 0);
                    L.n_int = S.word(slot, S.Q_GEN, 1);
                    L.m_ray = (int)S.word(slot, S.Q_GEN, 2);
                }
                if (LM) {
                    const float4 g = S.at(slot, S.Q_LM);
                    L.cx = __float_as_int(c.y);
                    L.cy = __float_as_int(d.w);
                    L.idx = g.x; L.idy = g.y; L.idz = g.z;
                    L.cz = __float_as_int(g.w);
                }
                L.state = which == S_COMP && (jf & JF_RAYLEIGH) ? S_RAY : which;
            }
        }
        if (which == S_GATHER) {
            if (slot >= 0) {
                int ie; float f;
                interp_index(L.e, P.e0, P.inv_de, P.n_e, ie, f);
                float r[NM], co[NM];
                coef_kind<NM>(P, 0, ie, f, r);
                coef_kind<NM>(P, 1, ie, f, co);
#pragma unroll
                for (int m = 0; m < NM; ++m) { L.cf(1, m) = r[m]; L.cf(2, m) = co[m]; }
                L.tot = reinterpret_cast<const float*>(&S.at(slot, 4));
                L.gather(P, ev);
            }
            tally(GDRR_ST_VIRTUAL, L.state == S_FLY);
            tally(GDRR_ST_PHOTO, ev.has(GDRR_ST_PHOTO));
            // the interaction waits for its own full warp; a virtual collision draws
            // its next flight here (through the interactions' list, where that is a
            // full warp's, 2 mm torsos took 1 % longer with cells of 4 mm, 4 % with 8
            // and 25 % with 128)
            const bool hit = L.state == S_RAY || L.state == S_COMP;
            const unsigned mI = __ballot_sync(FULL, hit);
            if (hit) {
                S.word(slot, 2, 3) = jf | (L.state == S_RAY ? JF_RAYLEIGH : 0u);
                if (GEN) S.word(slot, S.Q_GEN, 2) = (uint32_t)L.m_ray;
                qI[nI + __popc(mI & below)] = (uint8_t)slot;
            }
            nI += __popc(mI);
            add(A_GATHER, (unsigned)n);
        } else if (which == S_COMP) {
            jf &= ~JF_RAYLEIGH;
            if (slot >= 0) {
                const uint32_t b0 = L.rs.blk;
                L.need_e = false;
                L.interact(P, ev);
                limit += L.rs.blk - b0;
                fresh = L.need_e;
                jf |= JF_SCATTERED;
            }
            tally(GDRR_ST_RAYLEIGH, ev.has(GDRR_ST_RAYLEIGH));
            tally(GDRR_ST_COMPTON, ev.has(GDRR_ST_COMPTON));
            tally(GDRR_ST_CUTOFF, ev.has(GDRR_ST_CUTOFF));
        } else {
            tally(A_ESC, L.state == S_ESC);
            if (L.state == S_ESC) L.escape(P, ev, true);
            tally(GDRR_ST_TALLY_PRIMARY, ev.has(GDRR_ST_TALLY_PRIMARY));
            tally(GDRR_ST_TALLY_SCATTER, ev.has(GDRR_ST_TALLY_SCATTER));
            tally(GDRR_ST_MISS, ev.has(GDRR_ST_MISS));
            unsigned need = exhausted ? 0u : __ballot_sync(FULL, slot >= 0);
            while (need) {
                unsigned long long first = next;
                if (first >= end) {
                    if (lane == 0) first = atomicAdd(P.counter, (unsigned long long)chunk);
                    first = __shfl_sync(FULL, first, 0);
                    if (first >= P.total) { exhausted = true; break; }
                    __syncwarp();
                    if (lane == 0) end = min(first + chunk, (unsigned long long)P.total);
                    __syncwarp();
                }
                const unsigned take = (unsigned)min((unsigned long long)__popc(need), end - first);
                const unsigned rank = (unsigned)__popc(need & below);
                ev.m = 0u;
                if (((need >> lane) & 1u) && rank < take) L.start(P, first + rank, ev);
                add(GDRR_ST_HISTORIES, take);
                tally(GDRR_ST_TALLY_PRIMARY, ev.has(GDRR_ST_TALLY_PRIMARY));
                tally(GDRR_ST_MISS, ev.has(GDRR_ST_MISS));
                __syncwarp();
                if (lane == 0) next = first + take;
                __syncwarp();
                need = __ballot_sync(FULL, slot >= 0 && L.state != S_FLY);
            }
            if (L.state == S_FLY) {
                limit = L.rs.blk + (uint32_t)P.max_steps;
                jf = (uint32_t)L.job;
                fresh = true;
            }
        }
        if (LM) {
            ev.m = 0u;
            const bool draw = L.state == S_FLY;
            if (draw) {
                L.nsteps = L.rs.blk + (uint32_t)P.max_steps - limit;
                L.lm_prepare(P, ev);
            }
            tally(GDRR_ST_STEP_LIMIT, ev.has(GDRR_ST_STEP_LIMIT));
            tally(GDRR_ST_STEPS, draw && L.state == S_FLY);
        }
        // photons that fly on go back to their slot with the next flight's words;
        // ended histories (not those that found no successor) to the last list
        const bool on = L.state == S_FLY;
        const bool gone = slot >= 0 && L.state == S_DEAD && (which != S_ESC || fresh);
        if (on) {
            if (fresh) {
                float t[NM], mumax;
                energy_totals<NM>(P, L.e, t, mumax);
                S.set_totals(slot, t);
                c.x = mumax;
                c.y = 1.0f / mumax;
            }
            uint32_t wy = 0;
            if constexpr (LM) {
                c.x = L.tau;
                c.y = __int_as_float(L.cx);
                wy = (uint32_t)L.cy;
                S.at(slot, S.Q_LM) = make_float4(L.idx, L.idy, L.idz, __int_as_float(L.cz));
            } else {
                const uint4 w = flight_block(L.rs.blk, flight_keys(L.rs.angle, L.rs.hlo, L.rs.hhi, P.rk), P.rk);
                L.tg = -log_uniform((w.x >> 8) + 1u);
                wy = w.y;
                if (GEN) L.wz = w.z;
            }
            S.at(slot, 0) = make_float4(L.px, L.py, L.pz, L.tg);
            S.at(slot, 1) = make_float4(L.dx, L.dy, L.dz, L.e);
            S.at(slot, 2) = make_float4(c.x, c.y, __uint_as_float(L.rs.hlo), __uint_as_float(jf));
            S.at(slot, 3) = make_float4(__uint_as_float(L.rs.blk), __uint_as_float(limit), __uint_as_float(L.rs.hhi),
                                        __uint_as_float(wy));
            if (GEN) { S.word(slot, S.Q_GEN, 0) = L.wz; S.word(slot, S.Q_GEN, 1) = L.n_int; }
        }
        if (gone) S.word(slot, 2, 3) = JF_DEAD;
        const unsigned mR = __ballot_sync(FULL, on), mE = __ballot_sync(FULL, gone);
        if (on) qR[nR + __popc(mR & below)] = (uint8_t)slot;
        if (gone) qE[nE + __popc(mE & below)] = (uint8_t)slot;
        nR += __popc(mR);
        nE += __popc(mE);
        __syncwarp();
    }

    // the flights that the cells (or the nearest voxel) decided stopped neither
    // at a tentative collision nor outside the box
    __syncwarp();
    if (!LM && lane == 0) {
        const unsigned long long inl = acc[GDRR_ST_STEPS] - acc[A_GATHER] - acc[A_ESC];
        acc[GDRR_ST_VIRTUAL] += inl;
        if (!(GEN && (P.nearest_voxel || P.in_place))) acc[GDRR_ST_CELL_SKIPS] += inl;
    }
    __syncwarp();
    if (lane < GDRR_NSTATS && acc[lane]) atomicAdd(&cnt[lane], acc[lane]);
    __syncthreads();
    for (int i = threadIdx.x; i < GDRR_NSTATS; i += WARP_BLOCK)
        if (cnt[i]) atomicAdd(P.stats + i, cnt[i]);
}

// Gather roofline probe: the transport's trilinear corner gather (same
// layout, same index arithmetic) at pseudo-random cells, with nothing else,
// so the memory system's ceiling for this access pattern can be measured.
__global__ void __launch_bounds__(256) gather_probe_kernel(const McParams P, uint64_t n_cells,
                                                         unsigned int* sink) {
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t nth = (uint64_t)gridDim.x * blockDim.x;
    float acc = 0.0f;
    for (uint64_t i = tid; i < n_cells; i += nth) {
        uint32_t h = (uint32_t)i * 0x9E3779B1u;
        h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12; h *= 0x297A2D39u; h ^= h >> 15;
        const uint32_t h2 = h * 0x85EBCA6Bu ^ (h >> 13);
        const uint32_t h3 = h2 * 0xC2B2AE35u ^ (h2 >> 16);
        const float fx = (float)(h & 0xffffu) * (1.0f / 65536.0f) * (float)P.nx - 0.5f;
        const float fy = (float)(h2 & 0xffffu) * (1.0f / 65536.0f) * (float)P.ny - 0.5f;
        const float fz = (float)(h3 & 0xffffu) * (1.0f / 65536.0f) * (float)P.nz - 0.5f;
        const int gx = (int)floorf(fx), gy = (int)floorf(fy), gz = (int)floorf(fz);
        const float tx = fx - (float)gx, ty = fy - (float)gy, tz = fz - (float)gz;
        const int x0 = min(max(gx, 0), P.nx - 1), x1 = min(max(gx + 1, 0), P.nx - 1);
        const int y0 = min(max(gy, 0), P.ny - 1), y1 = min(max(gy + 1, 0), P.ny - 1);
        const int z0 = min(max(gz, 0), P.nz - 1), z1 = min(max(gz + 1, 0), P.nz - 1);
        const float wxy[4] = {(1.0f - tx) * (1.0f - ty), tx * (1.0f - ty), (1.0f - tx) * ty, tx * ty};
        const int bx[2] = {brick_x(x0), brick_x(x1)};
        const int by[2] = {brick_y(y0, P.bsy), brick_y(y1, P.bsy)};
        const int bz[2] = {brick_z(z0, P.bsz), brick_z(z1, P.bsz)};
        const int rows[4] = {by[0] + bz[0], by[1] + bz[0], by[0] + bz[1], by[1] + bz[1]};
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint2 vx = __ldg(P.vox + rows[c >> 1] + bx[c & 1]);
            acc = acc + (wxy[c & 3] * ((c >> 2) ? tz : 1.0f - tz)) * __uint_as_float(vx.x) * (float)(vx.y + 1u);
        }
    }
    if (acc == -1.0f) atomicAdd(sink, 1u);   // keeps the loads; never true for densities >= 0
}

__global__ void stream_words_kernel(const RoundKeys rk, uint32_t angle_index, uint64_t hid0, int n_hist,
                                    int n_blocks, uint32_t* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_hist) return;
    Stream rs;
    rs.init(angle_index, hid0 + (uint64_t)i);
    uint32_t* o = out + (size_t)i * 4 * n_blocks;
    for (int b = 0; b < n_blocks; ++b) {
        const uint4 w = rs.block(rk);
        o[4 * b] = w.x; o[4 * b + 1] = w.y; o[4 * b + 2] = w.z; o[4 * b + 3] = w.w;
    }
}

__global__ void flight_logs_kernel(uint32_t k0, int n, float* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = log_uniform(k0 + (uint32_t)i);
}

template <int NM>
constexpr size_t smem_bytes(int block) { return (size_t)3 * NM * block * sizeof(float); }

// Per-thread coefficient tables beyond 47 KB per block (8 materials at 512
// threads) need the kernel's dynamic shared-memory cap raised first.
template <int NM, bool GEN, bool LM>
cudaError_t launch_records_t(const McParams& p, int block, int per_sm_max, int n_sm, cudaStream_t s) {
    const size_t bytes = smem_bytes<NM>(block);
    cudaError_t e = cudaSuccess;
    if (smem_bytes<NM>(512) > 47 * 1024) e = allow_smem(mc_kernel<NM, GEN, LM>, smem_bytes<NM>(512));
    int per_sm = per_sm_max;
    if (e == cudaSuccess && per_sm <= 0)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mc_kernel<NM, GEN, LM>, block, bytes);
    if (e != cudaSuccess) return e;
    const int64_t useful = (int64_t)((p.total + 31) / 32 * 32 + block - 1) / block;
    const int64_t grid = std::min<int64_t>((int64_t)std::max(per_sm, 1) * n_sm, useful);
    mc_kernel<NM, GEN, LM><<<(int)std::max<int64_t>(grid, 1), block, bytes, s>>>(p);
    return cudaGetLastError();
}

// no cell test: none is wanted, or an axis has corners that corner_bits cannot count
inline bool without_cells(const McParams& p) { return !p.cells || std::max(p.nx, std::max(p.ny, p.nz)) >= 1 << 22; }

inline bool in_place(const McParams& p) {
    return p.lm ? lm_in_place(cell_edge(p.vox_mm, p.cshift))
                : without_cells(p) || coarse_in_place(cell_edge(p.vox_mm, p.cshift));
}

template <int NM, bool GEN, bool LM>
cudaError_t launch_warp_t(const McParams& p, int n_pool, int warps_max, int n_sm, cudaStream_t s) {
    if (n_pool <= 0) n_pool = default_pool(NM, GEN, LM);
    const size_t bytes = pool_bytes(n_pool, NM, GEN, LM) * POOL_WARPS;
    cudaError_t e = allow_smem(mc_warp_kernel<NM, GEN, LM>, pool_bytes(POOL_MAX, NM, GEN, LM) * POOL_WARPS);
    int per_sm = 0;
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mc_warp_kernel<NM, GEN, LM>, WARP_BLOCK, bytes);
    if (e != cudaSuccess) return e;
    if (per_sm <= 0) return cudaErrorInvalidConfiguration;
    constexpr int WPB = POOL_WARPS;
    if (warps_max > 0) per_sm = std::max(1, std::min(per_sm, (warps_max + WPB - 1) / WPB));
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((int64_t)per_sm * n_sm, (int64_t)((p.total + WPB - 1) / WPB)));
    const int64_t warps = grid * WPB;
    // a small launch spreads over every warp: fewer photons per warp, smaller claims
    const uint64_t share = (p.total + warps - 1) / warps;
    const int n_use = (int)std::min<uint64_t>((uint64_t)n_pool, share);
    const unsigned chunk = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)p.chunk, share / 4 + 1));
    McParams q = p;
    q.in_place = in_place(p);
    if (!LM && without_cells(p)) {
        q.cells = q.open_cell;
        q.cshift = 30;
        q.csx = q.csy = 0;
    }
    const uint32_t c = 0x4b000000u >> q.cshift;
    const uint32_t cell0 = c + (uint32_t)q.csx * (c + (uint32_t)q.csy * c);
    mc_warp_kernel<NM, GEN, LM><<<(int)grid, WARP_BLOCK, bytes, s>>>(q, n_pool, n_use, chunk, cell0);
    return cudaGetLastError();
}

template <bool GEN, bool LM>
cudaError_t launch_nm(const McParams& p, bool records, int block, int n_pool, int limit, int n_sm, cudaStream_t s) {
    if (records) {
        if (p.n_mat <= 2) return launch_records_t<2, GEN, LM>(p, block, limit, n_sm, s);
        if (p.n_mat <= 4) return launch_records_t<4, GEN, LM>(p, block, limit, n_sm, s);
        return launch_records_t<8, GEN, LM>(p, block, limit, n_sm, s);
    }
    const int warps = limit * block / 32;
    if (p.n_mat <= 2) return launch_warp_t<2, GEN, LM>(p, n_pool, warps, n_sm, s);
    if (p.n_mat <= 4) return launch_warp_t<4, GEN, LM>(p, n_pool, warps, n_sm, s);
    return launch_warp_t<8, GEN, LM>(p, n_pool, warps, n_sm, s);
}

}  // namespace

// photons: photons per lane in a warp's pool (1 .. 3), or <= 0 for the default
cudaError_t launch_mc(const McParams& p, int block, int blocks_per_sm, int photons, bool records, int n_sm,
                      cudaStream_t s) {
    if (p.lm && !p.cells) return cudaErrorInvalidValue;   // the local majorants are the cell bounds
    // the mixture in the flight or walk is the general form's alone, which has the
    // registers for it: 1e8 histories of the 2 mm torso without a cell test took
    // 209 ms by way of the gather service (156 with one photon per lane), so 134
    const bool gen = p.nearest_voxel != 0 || p.scatter_filter != 0 || p.ray_ff != 0 || (!records && in_place(p));
    const int n_pool = photons > 0 ? 32 * photons : 0;
    if (p.lm) return gen ? launch_nm<true, true>(p, records, block, n_pool, blocks_per_sm, n_sm, s)
                         : launch_nm<false, true>(p, records, block, n_pool, blocks_per_sm, n_sm, s);
    return gen ? launch_nm<true, false>(p, records, block, n_pool, blocks_per_sm, n_sm, s)
               : launch_nm<false, false>(p, records, block, n_pool, blocks_per_sm, n_sm, s);
}

cudaError_t launch_gather_probe(const McParams& p, uint64_t n_cells, int grid, unsigned int* sink, cudaStream_t s) {
    gather_probe_kernel<<<grid, 256, 0, s>>>(p, n_cells, sink);
    return cudaGetLastError();
}

cudaError_t launch_stream_words(uint64_t seed, uint32_t angle_index, uint64_t hid0, int n_hist, int n_blocks,
                                uint32_t* out, cudaStream_t s) {
    if (n_hist <= 0) return cudaSuccess;
    stream_words_kernel<<<(n_hist + 127) / 128, 128, 0, s>>>(round_keys(seed), angle_index, hid0, n_hist, n_blocks,
                                                             out);
    return cudaGetLastError();
}

cudaError_t launch_flight_logs(uint32_t k0, int n, float* out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    flight_logs_kernel<<<(n + 255) / 256, 256, 0, s>>>(k0, n, out);
    return cudaGetLastError();
}

}  // namespace gdrr
