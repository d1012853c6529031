// npp_device.cuh -- device-side building blocks of the planner library:
// the counter-based parameter sampler, the per-handle constants and the
// kernel argument blocks shared by the kernels and their launchers.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/npp.h"

namespace npp {

constexpr int NIN = 8;               // network inputs (features)
constexpr uint32_t FULL = 0xffffffffu;

// Constants derived once per handle from npp_config (FP32, device side).
struct DevCfg {
    float delta_max, r_rate;         // steering limit, rate limit per step (normalised)
    float lrL, iL;                   // l_r / (l_f + l_r), 1 / (l_f + l_r)
    float umid, uhalf;               // u = umid + uhalf a1
    float Ts;
    float ihl, ihw, c_off;           // 1/half_len, 1/half_wid, centre offset
    float idxi, ideta, idphi, idv;   // 1 / feature normalisation constants
    float w_pos, w_phi, w_v, w_effort;
    int body_frame;                  // goal offsets of the features in the frame at t+h
    int vlim;                        // speed limits on: discard at the first h >= 1 outside
    float v_lo, v_hi;                // [v_lo, v_hi]
};

// The device constants of a validated configuration (host side).
inline DevCfg devcfg_from(const npp_config& cfg)
{
    DevCfg d;
    const double L = (double)cfg.lf + cfg.lr;
    d.delta_max = cfg.delta_max;
    d.r_rate = (float)((double)cfg.delta_rate_max * cfg.Ts / cfg.delta_max);
    d.lrL = (float)(cfg.lr / L);
    d.iL = (float)(1.0 / L);
    d.umid = (float)(0.5 * ((double)cfg.u_min + cfg.u_max));
    d.uhalf = (float)(0.5 * ((double)cfg.u_max - cfg.u_min));
    d.Ts = cfg.Ts;
    d.ihl = (float)(1.0 / cfg.half_len);
    d.ihw = (float)(1.0 / cfg.half_wid);
    d.c_off = cfg.c_off;
    d.idxi = (float)(1.0 / cfg.dxi_n);
    d.ideta = (float)(1.0 / cfg.deta_n);
    d.idphi = (float)(1.0 / cfg.dphi_n);
    d.idv = (float)(1.0 / cfg.dv_n);
    d.w_pos = cfg.w_pos; d.w_phi = cfg.w_phi; d.w_v = cfg.w_v; d.w_effort = cfg.w_effort;
    d.body_frame = cfg.feature_frame;
    d.vlim = cfg.v_limits;
    d.v_lo = cfg.v_min;
    d.v_hi = cfg.v_max;
    return d;
}

// Range check of the variant fields of a configuration; null when valid.
inline const char* variant_error(const npp_config& cfg)
{
    if (cfg.feature_frame != 0 && cfg.feature_frame != 1) return "feature_frame is 0 or 1";
    if (cfg.v_limits != 0 && cfg.v_limits != 1) return "v_limits is 0 or 1";
    if (cfg.v_limits == 1 && !(std::isfinite(cfg.v_min) && std::isfinite(cfg.v_max) && cfg.v_min <= cfg.v_max))
        return "v_limits needs finite v_min <= v_max";
    return nullptr;
}

// Range check of the vehicle, feature and cost constants and the variant
// fields of a configuration (not the network shape, not the capacities);
// null when valid.  Every entry point that takes a configuration uses it.
inline const char* config_error(const npp_config& cfg)
{
    const float* f = &cfg.lf;                // the 18 float constants lf .. w_effort
    for (int i = 0; i < 18; ++i)
        if (!std::isfinite(f[i])) return "config has a non-finite constant";
    if (!(cfg.lf + cfg.lr > 0.f) || !(cfg.lr >= 0.f) || !(cfg.delta_max > 0.f) ||
        !(cfg.delta_rate_max > 0.f) || !(cfg.u_max >= cfg.u_min) || !(cfg.Ts > 0.f) ||
        !(cfg.half_len > 0.f) || !(cfg.half_wid > 0.f) || !(cfg.dxi_n > 0.f) ||
        !(cfg.deta_n > 0.f) || !(cfg.dphi_n > 0.f) || !(cfg.dv_n > 0.f))
        return "config constant out of range";
    return variant_error(cfg);
}

// ------------------------------------------------------------------ packed FP32
// Two FP32 values in one 64-bit register pair, for the packed FP32x2
// instructions: each half is rounded exactly as the scalar instruction
// rounds it.
__device__ __forceinline__ unsigned long long f2_pack(float lo, float hi)
{
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float2 f2_unpack(unsigned long long v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b,
                                                     unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long f2_mul(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long f2_both(float x) { return f2_pack(x, x); }

// ------------------------------------------------------------------ sampler
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw: "Parallel random numbers: as
// easy as 1, 2, 3", SC'11): ten rounds of two 32x32->64 multiplies with the
// published multipliers, key bumped by the published Weyl constants.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        const uint64_t p0 = (uint64_t)0xD2511F53u * c.x, p1 = (uint64_t)0xCD9E8D57u * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ k0, (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ k1,
                       (uint32_t)p0);
    }
    return c;
}

__device__ __forceinline__ float sfu_rcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sfu_rsqrt(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The two Box-Muller pairs of four Philox words (the FP32 sampler
// specification), evaluated side by side as the halves of packed FP32x2
// instructions:
//
//   u     = (2 (w >> 9) + 1) 2^-24, from words x and z
//   ln u  u = 2^e f with f in [sqrt(1/2), sqrt(2)), ln f = 2 atanh(s),
//         s = (f - 1) / (f + 1), odd Taylor terms up to s^11, Cody-Waite
//         split of ln 2
//   r     = sqrt(-2 ln u)
//   angle 2 pi K 2^-24, K = 2 (w >> 9) + 1, from words y and w:
//         quarter-turn reduction in integers (exact), Taylor polynomials of
//         degree 9 / 10 on |x| <= pi/4
//
// Every operation rounds to nearest once, so the values are reproducible bit
// for bit.  The quotient s and the root r are the correctly rounded ones of
// the specification, computed without a branch: an approximate reciprocal
// (reciprocal root), the product with it, and one correction by the exact
// fma residual (Markstein, "Computation of elementary functions on the IBM
// RISC System/6000 processor", IBM J. Res. Dev. 34, 1990).  The arguments
// are the 2^23 values of u; tests/test_gpu_sampler.py compares the results with
// the IEEE quotient and root on 98 % of them.
// Integer-to-float conversions are exact bit constructions (1.m minus a
// constant) except the exponent's.
//
// Bound: instruction issue -- parameter generation is 20-30 % of the
// rollout kernels' instructions.  Per quad about 135 instead of 210
// instructions (two independent scalar pairs with the IEEE division and
// root sequences and their range-check branches).  Plan steps measured on
// GB300: course (N = 16384, T = 40, width 32) 221 -> 198 us, large (N =
// 65536, T = 100, width 64) 2.61 -> 2.37 ms.
__device__ __forceinline__ float4 spec_normal_quad(const uint4& w)
{
    typedef unsigned long long f2;
    // u: 1.m - (1 - 2^-24) is exact
    const f2 u = f2_add(f2_pack(__uint_as_float((w.x >> 9) | 0x3F800000u),
                                __uint_as_float((w.z >> 9) | 0x3F800000u)), f2_both(-0x1.fffffep-1f));
    const float2 uu = f2_unpack(u);
    // e and f: the bits from those of sqrt(1/2) upwards, e in the exponent's place
    const uint32_t b0 = __float_as_uint(uu.x), b1 = __float_as_uint(uu.y);
    const uint32_t e0 = (b0 - 0x3F3504F4u) & 0xFF800000u, e1 = (b1 - 0x3F3504F4u) & 0xFF800000u;
    const f2 f = f2_pack(__uint_as_float(b0 - e0), __uint_as_float(b1 - e1));
    const f2 ef = f2_pack(__int2float_rn((int)e0), __int2float_rn((int)e1));   // e 2^23
    // -s: the negated reciprocal costs nothing (an operand modifier) and the
    // fma residual needs one of its factors negated; P's signs undo it
    const f2 num = f2_add(f, f2_both(-1.0f)), den = f2_add(f, f2_both(1.0f));
    const float2 dd = f2_unpack(den);
    const f2 rd = f2_pack(sfu_rcp(-dd.x), sfu_rcp(-dd.y));
    const f2 q = f2_mul(num, rd);
    const f2 s = f2_fma(f2_fma(den, q, num), rd, q);
    const f2 z = f2_mul(s, s);
    f2 p = f2_fma(z, f2_both(-0x1.745d18p-3f), f2_both(-0x1.c71c72p-3f));       // 2/11, 2/9
    p = f2_fma(z, p, f2_both(-0x1.24924ap-2f));                                   // 2/7
    p = f2_fma(z, p, f2_both(-0x1.99999ap-2f));                                   // 2/5
    p = f2_fma(z, p, f2_both(-0x1.555556p-1f));                                   // 2/3
    const f2 lnf = f2_fma(f2_mul(s, z), p, f2_mul(s, f2_both(-2.0f)));
    // ln 2 in two parts, scaled by 2^-23 for e 2^23
    const f2 ln = f2_fma(ef, f2_both(0x1.62e400p-24f), f2_fma(ef, f2_both(0x1.7f7d1cp-43f), lnf));
    // -r from x = 2 ln u = -r^2
    const f2 x = f2_add(ln, ln);
    const float2 xx = f2_unpack(x);
    const f2 y = f2_pack(sfu_rsqrt(-xx.x), sfu_rsqrt(-xx.y));
    const f2 g = f2_mul(x, y);
    const f2 r = f2_fma(f2_fma(g, g, x), f2_mul(y, f2_both(0.5f)), g);
    // angle: t = (w + an eighth turn) counts quarter turns in its top bits;
    // the remainder as 1.m - (1.5 - 2^-22) = k 2^-22 is exact
    const uint32_t t0 = w.y + 0x20000000u, t1 = w.w + 0x20000000u;
    const f2 k = f2_add(f2_pack(__uint_as_float(((t0 >> 7) & 0x007FFFFCu) | 0x3F800000u),
                                __uint_as_float(((t1 >> 7) & 0x007FFFFCu) | 0x3F800000u)),
                        f2_both(-(1.5f - 0x1p-22f)));
    const f2 a = f2_mul(k, f2_both(0x1.921fb6p0f));
    const f2 v = f2_mul(a, a);
    f2 ps = f2_fma(v, f2_both(0x1.71de3ap-19f), f2_both(-0x1.a01a02p-13f));
    ps = f2_fma(v, ps, f2_both(0x1.111112p-7f));
    ps = f2_fma(v, ps, f2_both(-0x1.555556p-3f));
    const f2 sx = f2_fma(f2_mul(a, v), ps, a);
    f2 pc = f2_fma(v, f2_both(-0x1.27e4fcp-22f), f2_both(0x1.a01a02p-16f));
    pc = f2_fma(v, pc, f2_both(-0x1.6c16c2p-10f));
    pc = f2_fma(v, pc, f2_both(0x1.555556p-5f));
    pc = f2_fma(v, pc, f2_both(-0.5f));
    const f2 cx = f2_fma(v, pc, f2_both(1.0f));
    // times -r before the quadrant's swap and signs (a sign flip is exact)
    const float2 rs = f2_unpack(f2_mul(r, sx)), rc = f2_unpack(f2_mul(r, cx));
    const bool o0 = (t0 >> 30) & 1u, o1 = (t1 >> 30) & 1u;
    float4 n;
    n.x = __uint_as_float(__float_as_uint(o0 ? rs.x : rc.x) ^ (~(t0 ^ (t0 << 1)) & 0x80000000u));
    n.y = __uint_as_float(__float_as_uint(o0 ? rc.x : rs.x) ^ (~t0 & 0x80000000u));
    n.z = __uint_as_float(__float_as_uint(o1 ? rs.y : rc.y) ^ (~(t1 ^ (t1 << 1)) & 0x80000000u));
    n.w = __uint_as_float(__float_as_uint(o1 ? rc.y : rs.y) ^ (~t1 & 0x80000000u));
    return n;
}

struct SamplerKey {
    uint32_t k0, k1, t_index, stream_id;
};

// theta_n[4q .. 4q+3]
__device__ __forceinline__ float4 sample_quad(const SamplerKey& key, uint32_t q, uint32_t n)
{
    const uint4 w = philox4x32_10(make_uint4(q, n, key.t_index, key.stream_id), key.k0, key.k1);
    return spec_normal_quad(w);
}

// theta_n[i], theta_n[i+1] for even i (one Box-Muller pair of its quad)
__device__ __forceinline__ float2 sample_pair(const SamplerKey& key, uint32_t i, uint32_t n)
{
    const uint4 w = philox4x32_10(make_uint4(i >> 2, n, key.t_index, key.stream_id), key.k0, key.k1);
    const float4 v = spec_normal_quad(w);
    return (i & 2u) ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
}

// Gaussian sampling proposal of a plan step: samples n < n_prop take
// theta_i = fma(sigma_i, eps_i, mu_i) with eps the normals of stream
// `stream` (1 for the learned proposal; the restart rounds of the hill
// climb use 1, 2, ...) rounded once to FP32; the others are the isotropic
// samples.  mu and sigma hold n_theta FP32 values.
struct Proposal {
    const float* mu;
    const float* sigma;
    int n_prop;
    uint32_t stream;      // Philox stream of the proposal's normals (1 unless set)
};

__device__ __forceinline__ bool proposal_sample(const Proposal& p, uint32_t n)
{
    return p.mu != nullptr && (long long)n < (long long)p.n_prop;
}

// four values from index i on (a multiple of 4) of an array that may start at
// any 4-byte boundary (vec: it starts at a 16-byte one)
__device__ __forceinline__ float4 load_quad(const float* p, int i, bool vec)
{
    if (vec) return *reinterpret_cast<const float4*>(p + i);
    return make_float4(p[i], p[i + 1], p[i + 2], p[i + 3]);
}

// theta_n[4q .. 4q+3] of a plan step with proposal p (all four indices
// below n_theta).  mu and sigma are read before the sampler's arithmetic,
// which hides the reads (a rolled loop of quads has nothing else to).
__device__ __forceinline__ float4 sample_quad_mixed(const SamplerKey& key, const Proposal& p, uint32_t q,
                                                    uint32_t n)
{
    if (!proposal_sample(p, n)) return sample_quad(key, q, n);
    SamplerKey k1 = key;
    k1.stream_id = p.stream;
    const bool vec = ((reinterpret_cast<uintptr_t>(p.mu) | reinterpret_cast<uintptr_t>(p.sigma)) & 15u) == 0;
    const float4 s = load_quad(p.sigma, 4 * (int)q, vec), m = load_quad(p.mu, 4 * (int)q, vec);
    const float4 e = sample_quad(k1, q, n);
    return make_float4(fmaf(s.x, e.x, m.x), fmaf(s.y, e.y, m.y), fmaf(s.z, e.z, m.z), fmaf(s.w, e.w, m.w));
}

// theta_n[i], theta_n[i+1] for even i
__device__ __forceinline__ float2 sample_pair_mixed(const SamplerKey& key, const Proposal& p, uint32_t i,
                                                    uint32_t n)
{
    if (!proposal_sample(p, n)) return sample_pair(key, i, n);
    SamplerKey k1 = key;
    k1.stream_id = p.stream;
    const float2 s = make_float2(p.sigma[i], p.sigma[i + 1]), m = make_float2(p.mu[i], p.mu[i + 1]);
    const float2 e = sample_pair(k1, i, n);
    return make_float2(fmaf(s.x, e.x, m.x), fmaf(s.y, e.y, m.y));
}

// Obstacle point o = (x, y, vx, vy) in the EV frame of the plan step (origin
// (x0, y0), heading with sine s0 and cosine c0), rounding fixed by explicit
// fmas so every collision path sees the same FP32 positions.
__device__ __forceinline__ void ev_point(const float4& o, float x0, float y0, float s0, float c0,
                                         float& px, float& py, float& vx, float& vy)
{
    const float dx = o.x - x0, dy = o.y - y0;
    px = fmaf(c0, dx, __fmul_rn(s0, dy));
    py = fmaf(-s0, dx, __fmul_rn(c0, dy));
    vx = fmaf(c0, o.z, __fmul_rn(s0, o.w));
    vy = fmaf(-s0, o.z, __fmul_rn(c0, o.w));
}

// theta[4q .. 4q+3] where the quad may run past n_theta (the proposal
// arrays hold exactly n_theta values)
__device__ __forceinline__ float4 sample_quad_mixed_tail(const SamplerKey& key, const Proposal& p, uint32_t q,
                                                         uint32_t n, int n_theta)
{
    if (4 * (int)q + 3 < n_theta || !proposal_sample(p, n)) return sample_quad_mixed(key, p, q, n);
    SamplerKey k1 = key;
    k1.stream_id = p.stream;
    const float4 e = sample_quad(k1, q, n);
    const float ev[4] = { e.x, e.y, e.z, e.w };
    float r[4] = { 0.f, 0.f, 0.f, 0.f };
    for (int j = 0; j < 4 && 4 * (int)q + j < n_theta; ++j) {
        const int i = 4 * (int)q + j;
        r[j] = fmaf(p.sigma[i], ev[j], p.mu[i]);
    }
    return make_float4(r[0], r[1], r[2], r[3]);
}

// ------------------------------------------------------------------ spatial bins
// Per-step grids of the binned collision check: for step h, cell_start[h]
// [BIN_DIM^2 + 1 entries, stride BIN_CS_STRIDE] indexes the points of
// step h sorted by cell, pts + h M (for the check with a step's grid in shared
// memory, 16-bit entries in the same place).  A query box within `reach` of a
// state spans at most five cells per axis.
constexpr int BIN_DIM = 128;
constexpr int BIN_NCELL = BIN_DIM * BIN_DIM;
constexpr int BIN_CS_STRIDE = BIN_NCELL + 4;    // 16-byte multiple: the float2 points that follow stay aligned

struct BinView {
    float x0;              // lower-left corner of the grid (EV frame, both axes)
    float inv_cell;
    float reach;           // radius around the reference point that holds the vehicle, plus a margin
    float cx, cy, hl, hw;  // a box that holds it too, in its own frame: centre, half extents plus the margin
    const int* cell_start; // null: no grids
    const float2* pts;
    int M;
};

// General footprint: the union of convex pieces, each the intersection of
// half-planes n . q < b in the vehicle's frame (q relative to the reference
// point, x along the heading), faces of one piece consecutive, w = 1 on the
// last face of a piece.
constexpr int FP_MAX_FACES = 64;
constexpr int FP_MAX_PIECES = 16;
struct PolyView {
    const float4* faces;   // [n_faces] (nx, ny, b, last) with |n| = 1
    int n_faces;           // 0: the rectangle
    int brute;             // 1: every point each step (no grid cells)
    float cx, cy, hl, hw;  // a box holding the footprint in its frame: centre, half extents plus a margin
};

__device__ __forceinline__ int bin_cell(float x, const BinView& g)
{
    const float f = floorf((x - g.x0) * g.inv_cell);
    return (int)fminf(fmaxf(f, 0.0f), (float)(BIN_DIM - 1));
}

// The candidate points of a query box (half extents rx, ry around (x, y), at
// most the grid's reach) in one step's grid: the cells of the at most five
// cell rows it overlaps, each row's cells one contiguous run of the
// cell-sorted points.  Cells are at least half as wide as the reach, so the
// box spans at most five cells per axis; indices are clamped monotonically at
// the grid border, so every point that can lie in the box is a candidate.
constexpr int BIN_MAX_ROWS = 5;      // cell rows a query can span (cells >= half the reach)
struct CandRows {
    int b[BIN_MAX_ROWS];             // first sorted point of each row's run
    int e[BIN_MAX_ROWS];             // candidates before the end of each run (inclusive prefix)
    int total;
    // index (into the step's sorted points) of candidate k < total
    __device__ __forceinline__ int index(int k) const
    {
        int i = b[0] + k;
#pragma unroll
        for (int r = 1; r < BIN_MAX_ROWS; ++r)
            if (k >= e[r - 1]) i = b[r] + (k - e[r - 1]);
        return i;
    }
};

struct QueryBox {
    float x, y, rx, ry;
};

__device__ __forceinline__ CandRows cand_rows(const int* __restrict__ cs, const BinView& g, const QueryBox& q)
{
    const int ix0 = bin_cell(q.x - q.rx, g), ix1 = bin_cell(q.x + q.rx, g);
    const int iy0 = bin_cell(q.y - q.ry, g), iy1 = bin_cell(q.y + q.ry, g);
    CandRows c;
    int acc = 0;
#pragma unroll
    for (int k = 0; k < BIN_MAX_ROWS; ++k) {
        int beg = 0, len = 0;
        if (iy0 + k <= iy1) {
            beg = cs[(iy0 + k) * BIN_DIM + ix0];
            len = cs[(iy0 + k) * BIN_DIM + ix1 + 1] - beg;
        }
        c.b[k] = beg;
        acc += len;
        c.e[k] = acc;
    }
    c.total = acc;
    return c;
}

// ------------------------------------------------------------------ rollout math
// FP32 functions of the rollout step built on the SFU's approximate base-2
// exponential, reciprocal, sine and cosine (PTX ex2/rcp/sin/cos .approx).
// Absolute errors (measured against the correctly rounded values on a dense
// grid of arguments, see the diagnostics entry point): tanh below 5e-7 for
// every finite x; tan below 2e-6 for |z| <= 1; sin/cos of the heading below
// 1e-6 for |phi| <= 1e3.

__device__ __forceinline__ float sfu_ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sfu_sin(float x)
{
    float y;
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sfu_cos(float x)
{
    float y;
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// tanh x = 1 - 2 / (e^{2x} + 1); e^{2x} = 2^{x * 2/ln 2}.  Saturates to
// +-1 (e^{2x} = inf gives 1, e^{2x} = 0 gives -1).
__device__ __forceinline__ float tanh_r(float x)
{
    const float e = sfu_ex2(x * 2.88539008177792681f);
    return fmaf(-2.0f, sfu_rcp(e + 1.0f), 1.0f);
}

// tanh_r of two values side by side (each rounding as above)
__device__ __forceinline__ void tanh_r2(float& x0, float& x1)
{
    const float2 t = f2_unpack(f2_mul(f2_pack(x0, x1), f2_both(2.88539008177792681f)));
    const float2 e = f2_unpack(f2_add(f2_pack(sfu_ex2(t.x), sfu_ex2(t.y)), f2_both(1.0f)));
    const float2 r = f2_unpack(f2_fma(f2_both(-2.0f), f2_pack(sfu_rcp(e.x), sfu_rcp(e.y)), f2_both(1.0f)));
    x0 = r.x;
    x1 = r.y;
}

// tan z = sin z / cos z for the steering angle (|z| <= delta_max < pi/2)
__device__ __forceinline__ float tan_r(float z)
{
    return sfu_sin(z) * sfu_rcp(sfu_cos(z));
}

// sin and cos of a heading: Cody-Waite reduction by 2 pi (two-part constant,
// 2 pi = TWO_PI_HI + TWO_PI_LO) to |r| <= pi, then the SFU on r
__device__ __forceinline__ void sincos_r(float phi, float& s, float& c)
{
    const float TWO_PI_HI = 6.28318548202514648f;      // float nearest 2 pi
    const float TWO_PI_LO = -1.74845553146951715e-7f;  // 2 pi - TWO_PI_HI
    const float k = rintf(phi * 0.159154943091895336f);
    float r = fmaf(-k, TWO_PI_HI, phi);
    r = fmaf(-k, TWO_PI_LO, r);
    s = sfu_sin(r);
    c = sfu_cos(r);
}

// ------------------------------------------------------------------ kernels
// State of a device-resident closed loop (Alg. 1 run inside a CUDA graph).
// The plan-step kernels read the planner's view of it; the advance kernel
// moves the simulated vehicle and the mission forward.
struct LoopDev {
    float x0, y0, phi0, v0, ap0, ap1;  // vehicle state at this sampling time (FP32 view)
    float gx, gy, gphi, gv;            // current goal setpoint
    uint32_t t_index;                  // sampling time (Philox counter word)
    int warm_valid;                    // the warm-start buffer holds theta*_{t-1}
    double px, py, pphi, pv;           // simulated vehicle (FP64)
    double cphi, sphi;                 // cosine and sine of pphi
    int waypoint, n_wp, done, t;
    int status, best_idx, n_infeasible;
    float best_cost;
    float eps[4];                      // completion tolerances (xi, eta, phi, v)
    // mission mode (reference path): space index, next stop setpoint, goal
    // setpoint index, range field (front, back, side), index search window,
    // points outside the range field hidden from the plan step
    int mission, idx, stop, goal_k, window, hide;
    float field[3];
};

// Per-step scalars of a plan step, from the arguments or from a LoopDev.
struct StepIn {
    float x0, y0, phi0, v0, ap0, ap1, gx, gy, gphi, gv;
    uint32_t t_index;
    bool warm_ok;
};

// blocks of 32 point pairs (64 points) holding M obstacle points in the
// brute-force checks' layout (XY entries of a block, then its V entries)
__host__ __device__ constexpr int pair_blocks(int M) { return (M + 63) / 64; }

struct RolloutArgs {
    DevCfg c;
    float x0, y0, phi0, v0, ap0, ap1;  // world-frame state and last controls
    float gx, gy, gphi, gv;            // world-frame goal
    const float4* obs;                 // [M] world frame (x, y, vx, vy)
    int M, N, T;
    SamplerKey key;
    const float* theta;                // explicit parameters [N][n_theta] or null
    const float* warm;                 // replaces sample 0 when non-null
    Proposal prop;                     // sampling proposal (mu null: isotropic only)
    float* costs;                      // [N] or null
    int* first_hit;                    // [N] or null
    float4* traj;                      // [T+1][N] EV frame (always written)
    float2* ctrl;                      // [T][N]
    float* jfree;                      // [N] cost of each sample if collision-free
    int* vfirst;                       // [N] first speed-violating step (-1 none), written by the
                                       // trajectory kernel when c.vlim; null otherwise
    unsigned long long* best_key;      // packed (class, cost, index) minimum
    unsigned long long* reset_key;     // the minimum, for the trajectory kernel to start (null: started elsewhere)
    unsigned* work;                    // work-queue counter of the persistent collision kernel
    int grid_collide;                  // persistent grid size
    int sm_count;                      // SMs of the device
    const LoopDev* dyn;                // when set, per-step scalars come from here
    int warm_force;                    // the warm start replaces sample 0 even before the loop's
                                       // first step (restart rounds: it is the incumbent)
    float4* pXY;                       // EV-frame point pairs in global memory when the points
                                       // exceed shared memory: 64 pair_blocks(M) entries, the
                                       // shared-memory staging's blocked layout
    unsigned* fault;                   // set when a bounded device wait gave up (read and
                                       // cleared by the winner epilogue), or null
    BinView bins;                      // per-step grids (binned and fused collision checks)
    unsigned long long* counts;        // measurement counters, or null: [0] candidate point tests
                                       // and [1] states checked by the binned check, [2] sample-steps
                                       // computed by the trajectory kernel
    // Step chunks (binned check, no per-sample records wanted): a
    // trajectory launch computes steps chunk_lo .. chunk_hi - 1 (states up to
    // chunk_hi), the check covers the states the chunk produced; chunk_hi 0:
    // the whole horizon in one launch each.  live_in (length *live_n_in)
    // lists the samples still collision-free before the chunk (null: all N);
    // the check appends the chunk's survivors to live_out, counting in
    // *live_n_out.  carry: [N] values carried between chunks.
    int chunk_lo, chunk_hi;
    const int* live_in;
    const int* live_n_in;
    int* live_out;
    int* live_n_out;
    float4* carry;
    PolyView poly;                     // general footprint (polygon checks)
    int* first;                        // [N] first colliding step so far (grid check; null: another check)
    int* done;                         // [GRID_MAX_CHUNKS] steps finished per sample chunk
};

__device__ __forceinline__ StepIn step_in(const RolloutArgs& a)
{
    StepIn s;
    if (a.dyn) {
        const LoopDev& d = *a.dyn;
        s.x0 = d.x0; s.y0 = d.y0; s.phi0 = d.phi0; s.v0 = d.v0; s.ap0 = d.ap0; s.ap1 = d.ap1;
        s.gx = d.gx; s.gy = d.gy; s.gphi = d.gphi; s.gv = d.gv;
        s.t_index = d.t_index;
        s.warm_ok = d.warm_valid != 0 || a.warm_force != 0;
    } else {
        s.x0 = a.x0; s.y0 = a.y0; s.phi0 = a.phi0; s.v0 = a.v0; s.ap0 = a.ap0; s.ap1 = a.ap1;
        s.gx = a.gx; s.gy = a.gy; s.gphi = a.gphi; s.gv = a.gv;
        s.t_index = a.key.t_index;
        s.warm_ok = true;
    }
    return s;
}

struct EpilogueArgs {
    float x0, y0, phi0;
    int N, T, n_theta;
    SamplerKey key;
    const float* warm;
    Proposal prop;
    const float4* traj;
    const float2* ctrl;
    const unsigned long long* best_key;
    void* best;                        // npp_best*
    float* params;
    float* controls;
    float* trajectory;
    const LoopDev* dyn;                // when set, x0, y0, phi0, t_index, warm validity from here
    int warm_force;                    // as RolloutArgs::warm_force
    unsigned* fault;                   // as RolloutArgs::fault: nonzero turns the result's status
                                       // into NPP_DEVICE_TIMEOUT (and is cleared), or null
};

// launchers: trajectory kernel per network width, one collision kernel
cudaError_t launch_traj_w16(const RolloutArgs& a, cudaStream_t s, int variant);
cudaError_t launch_traj_w32(const RolloutArgs& a, cudaStream_t s, int variant);
cudaError_t launch_traj_w64(const RolloutArgs& a, cudaStream_t s, int variant);
// trajectories with the binned collision check done window by window by
// the trajectory warps (a.bins set): each sample stops within one window
// of its first collision; writes costs, first hits, the key and the states
// and controls up to that window
cudaError_t launch_fused_w16(const RolloutArgs& a, cudaStream_t s, int variant);
cudaError_t launch_fused_w32(const RolloutArgs& a, cudaStream_t s, int variant);
cudaError_t launch_fused_w64(const RolloutArgs& a, cudaStream_t s, int variant);
cudaError_t launch_collide_resident(const RolloutArgs& a, cudaStream_t s, int variant);
cudaError_t launch_collide_states(const RolloutArgs& a, cudaStream_t s);   // one lane per state (few points)
cudaError_t launch_collide_global(const RolloutArgs& a, cudaStream_t s);
int collide_global_blocks_per_sm();
int collide_resident_blocks_per_sm(int M, int variant);
int collide_max_points(int smem_limit);
// collisions through per-step spatial binning of the points (any M): builds
// the grids in `workspace` (binned_workspace_bytes) and checks every sample
// against the points of the cells that the box around it overlaps
size_t binned_workspace_bytes(int max_T, int max_M);
cudaError_t build_bins(RolloutArgs& a, float half_len, float half_wid, float c_off, void* workspace,
                       cudaStream_t s);          // fills a.bins
// the rectangle's binned check with a step's grid in shared memory (M <=
// collide_grid_points()); the grid build starts `first` and `done`
constexpr int GRID_MAX_CHUNKS = 1024;
int collide_grid_points();
cudaError_t launch_collide_grid(const RolloutArgs& a, cudaStream_t s);
cudaError_t launch_count_grid(const RolloutArgs& a, cudaStream_t s);   // its work, after it
cudaError_t launch_collide_binned(const RolloutArgs& a, cudaStream_t s);
cudaError_t launch_collide_poly(const RolloutArgs& a, cudaStream_t s);     // every point (a.poly.brute)
// grids for a general footprint inside the disk of the given radius around
// the reference point and inside box (xmin, xmax, ymin, ymax) of its frame
cudaError_t build_bins_poly(RolloutArgs& a, double radius, const double box[4], void* workspace, cudaStream_t s);
cudaError_t launch_epilogue(const EpilogueArgs& e, cudaStream_t s);
void set_global_error(const char* msg);

}  // namespace npp
