// xy_device.cuh -- device-side building blocks shared by every stepping kernel.
//
// All arithmetic is written with explicit fmaf / __fmul_rn so that, with the
// library compiled under -fmad=false, every kernel that calls these functions
// produces bit-identical results for the same site and step (the plain, the
// strip and the resident steppers, the prime and full-step-velocity kernels,
// and the adjoint's recompute pass).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "xy_internal.h"

namespace xy {

// -------------------------------------------------------------------------
// The four sites of a quad as two pairs (0, 1), (2, 3).  sm_103a issues one
// FP32 instruction for a pair (fma.rn.f32x2 and its add and mul), each half
// rounded like the scalar instruction, so a pair costs one issue slot and the
// bits are those of the scalar code.  The steppers are bound by the issue of
// instructions, a third of which were FP32 adds and multiplies of whole quads: 82 per
// site-update in the one-step strip kernel and 70 in the first two-step kernel, 68
// and 44 now (the band kernel, at 58 % of the issue slots).
// -------------------------------------------------------------------------
struct P4 {
    float2 a, b;
};
__device__ __forceinline__ float2 splat2(float v) { return make_float2(v, v); }
__device__ __forceinline__ P4 p4(const float4& t) { return P4{make_float2(t.x, t.y), make_float2(t.z, t.w)}; }
__device__ __forceinline__ float4 f4(const P4& t) { return make_float4(t.a.x, t.a.y, t.b.x, t.b.y); }
__device__ __forceinline__ P4 add4(const P4& x, const P4& y) { return P4{__fadd2_rn(x.a, y.a), __fadd2_rn(x.b, y.b)}; }
__device__ __forceinline__ P4 mul4(const P4& x, const P4& y) { return P4{__fmul2_rn(x.a, y.a), __fmul2_rn(x.b, y.b)}; }
__device__ __forceinline__ P4 mul4(float k, const P4& y) { return P4{__fmul2_rn(splat2(k), y.a), __fmul2_rn(splat2(k), y.b)}; }
__device__ __forceinline__ P4 fma4(const P4& x, const P4& y, const P4& z)
{
    return P4{__ffma2_rn(x.a, y.a, z.a), __ffma2_rn(x.b, y.b, z.b)};
}
__device__ __forceinline__ P4 fma4(float k, const P4& y, const P4& z)
{
    return P4{__ffma2_rn(splat2(k), y.a, z.a), __ffma2_rn(splat2(k), y.b, z.b)};
}
__device__ __forceinline__ float p4get(const P4& v, int i)
{
    return i == 0 ? v.a.x : (i == 1 ? v.a.y : (i == 2 ? v.b.x : v.b.y));
}

// -------------------------------------------------------------------------
// Counter-based noise: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11).
// Counter = (quad, (config << 16) | replica, step lo32, (tag << 24) | step hi24),
// key = 64-bit seed.  One call gives the four Gaussians of four consecutive
// sites (a float4 of the state).
// -------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c.x;  // one wide multiply gives both halves
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c.z;
        const uint32_t lo0 = (uint32_t)p0, hi0 = (uint32_t)(p0 >> 32);
        const uint32_t lo1 = (uint32_t)p1, hi1 = (uint32_t)(p1 >> 32);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// The same function with the ten round keys precomputed (kernel parameters,
// so every XOR takes its key from the constant bank).
__device__ __forceinline__ uint4 philox4x32_10_rk(uint4 c, const PhiloxKeys& K)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c.x;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c.z;
        const uint32_t lo0 = (uint32_t)p0, hi0 = (uint32_t)(p0 >> 32);
        const uint32_t lo1 = (uint32_t)p1, hi1 = (uint32_t)(p1 >> 32);
        c = make_uint4(hi1 ^ c.y ^ K.k0[r], lo1, hi0 ^ c.w ^ K.k1[r], lo0);
    }
    return c;
}

__device__ __forceinline__ uint4 noise_counter(uint32_t quad, uint32_t cfg_rep, int64_t k, uint32_t tag)
{
    const uint64_t ku = (uint64_t)k;
    return make_uint4(quad, cfg_rep, (uint32_t)(ku & 0xFFFFFFFFu),
                      (tag << 24) | (uint32_t)((ku >> 32) & 0xFFFFFFu));
}

// Uniform (m + 1/2) 2^-23 in (0,1) from the top 23 bits of a word, exactly:
// the float 1 + m 2^-23 minus (1 - 2^-24) is exact by Sterbenz' lemma.  The
// bits of 1 + m 2^-23, 0x3F800000 | (x >> 9), are one funnel shift of 0x7F:x.
__device__ __forceinline__ float uniform01_plus(uint32_t x) { return __uint_as_float(__funnelshift_r(x, 0x7Fu, 9)); }
__device__ __forceinline__ float uniform01(uint32_t x) { return __fadd_rn(uniform01_plus(x), -0.99999994f); }

// Hardware log2 and reciprocal square root without the code that scales
// subnormal operands: the operands below are never subnormal (a uniform is at
// least 2^-24, and -2 ln u at least 1.2e-7), and for normal ones the results
// are those of __log2f and rsqrtf.
__device__ __forceinline__ float log2_normal(float x)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_normal(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Box-Muller (Box & Muller 1958) of two uniform pairs, scaled by the noise
// amplitude c: returns c*g0..c*g3 with g0 = r cos(2 pi u1), g1 = r sin(2 pi u1),
// g2 = r' cos(2 pi u3), g3 = r' sin(2 pi u3), r = sqrt(-2 ln u0),
// r' = sqrt(-2 ln u2).  The angle is shifted by -pi into the accurate range of
// the hardware sine, and the sign flip is folded into the radius.  The two
// Box-Muller pairs run as one packed pair.
__device__ __forceinline__ float4 gauss4_scaled(uint4 w, float c)
{
    const float kTwoPi = 6.28318530717958648f;
    const float kPi = 3.14159265358979324f;
    const float kM2Ln2 = -1.38629436111989061f;  // -2 ln 2
    const float2 ur = __fadd2_rn(make_float2(uniform01_plus(w.x), uniform01_plus(w.z)), splat2(-0.99999994f));
    const float2 ua = __fadd2_rn(make_float2(uniform01_plus(w.y), uniform01_plus(w.w)), splat2(-0.99999994f));
    const float2 t = __fmul2_rn(splat2(kM2Ln2), make_float2(log2_normal(ur.x), log2_normal(ur.y)));  // -2 ln u > 0
    const float2 r = __fmul2_rn(__fmul2_rn(t, make_float2(rsqrt_normal(t.x), rsqrt_normal(t.y))), splat2(-c));
    const float2 ang = __ffma2_rn(splat2(kTwoPi), ua, splat2(-kPi));
    float s0, c0, s1, c1;
    __sincosf(ang.x, &s0, &c0);
    __sincosf(ang.y, &s1, &c1);
    return make_float4(__fmul_rn(r.x, c0), __fmul_rn(r.x, s0), __fmul_rn(r.y, c1), __fmul_rn(r.y, s1));
}

// -------------------------------------------------------------------------
// State space: map an angle back into [-pi/2, pi/2) (Sec. III.D).
// -------------------------------------------------------------------------
// An angle already inside (-pi/2, pi/2) is returned as it is: one compare
// and a branch that is almost never taken, since a drift of dt v rarely
// crosses the cut (2.4 % more site-updates/s than reducing every angle).
// Any other value takes the full reduction.
__device__ __forceinline__ float wrap_angle_reduce(float t)
{
    const float kPi = 3.14159265358979324f;
    const float kInvPi = 0.318309886183790672f;
    const float kHalfPi = 1.57079632679489662f;
    const float n = floorf(fmaf(t, kInvPi, 0.5f));
    float r = fmaf(-kPi, n, t);
    r = (r >= kHalfPi) ? __fadd_rn(r, -kPi) : r;
    r = (r < -kHalfPi) ? __fadd_rn(r, kPi) : r;
    return r;
}

__device__ __forceinline__ float wrap_angle(float t)
{
    const float kHalfPi = 1.57079632679489662f;
    if (__builtin_expect(fabsf(t) < kHalfPi, 1)) return t;
    return wrap_angle_reduce(t);
}

// The same for the four angles of a quad: one test and one branch for all of
// them (a branch per angle took three instructions each).
__device__ __forceinline__ P4 wrap_angle4(P4 t)
{
    const float kHalfPi = 1.57079632679489662f;
    const float m = fmaxf(fmaxf(fabsf(t.a.x), fabsf(t.a.y)), fmaxf(fabsf(t.b.x), fabsf(t.b.y)));
    if (__builtin_expect(!(m < kHalfPi), 0)) {
        t.a = make_float2(wrap_angle(t.a.x), wrap_angle(t.a.y));
        t.b = make_float2(wrap_angle(t.b.x), wrap_angle(t.b.y));
    }
    return t;
}

// -------------------------------------------------------------------------
// Per-step constants of one configuration.
// -------------------------------------------------------------------------
struct StepConst {
    float c;        // half-kick noise amplitude (1/2) sqrt(2 eta T_k) sqrt(dt)
    float hdt;      // dt / 2
    float dt;
    float oma;      // 1 - eta dt / 2
    float inv1pa;   // 1 / (1 + eta dt / 2)
    float nqJx;     // -q J_par
    float nqJy;     // -q J_perp
    float hp;       // h p
    float q, p;
};

// Temperature at step k: piecewise linear through the knots, constant outside
// them, evaluated in FP32 from per-segment slopes (a few instructions per
// thread block or warp; never FP64 on the stepping path); or the nonlinear
// quench of order gamma.
__device__ __forceinline__ float temperature_at(const DevCfg& cf, int64_t k)
{
    if (cf.sched_kind == 1) {  // nonlinear quench (Sec. V), FP32
        const float t = (float)(k - cf.pw_kc);
        float eps = powf(__fmul_rn(fabsf(t), cf.pw_inv_tq), cf.pw_gamma);
        eps = t >= 0.f ? -eps : eps;
        eps = fminf(fmaxf(eps, cf.pw_ef), cf.pw_ei);
        return __fmul_rn(cf.pw_Tc, __fadd_rn(1.0f, eps));
    }
    if (cf.n_knots <= 1 || k <= cf.knot_step[0]) return cf.knot_Tf[0];
    for (int i = 0; i + 1 < cf.n_knots; ++i)
        if (k <= cf.knot_step[i + 1]) return fmaf(cf.slope_f[i], (float)(k - cf.knot_step[i]), cf.knot_Tf[i]);
    return cf.knot_Tf[cf.n_knots - 1];
}

// Half-kick noise amplitude c_k = (1/2) sqrt(2 eta T_k) sqrt(dt) (App. A.1).
__device__ __forceinline__ float noise_amp(const DevCfg& cf, int64_t k)
{
    const float T = temperature_at(cf, k);
    return __fmul_rn(cf.amp_pref, __fsqrt_rn(T > 0.f ? T : 0.f));
}

// Field schedule s(k) of the orthogonal quench: h_k = h s(k) (1 without one).
__device__ __forceinline__ float field_scale(const DevCfg& cf, int64_t k)
{
    if (cf.f_n_knots <= 1 || k <= cf.f_knot_step[0]) return cf.f_n_knots == 0 ? 1.0f : cf.f_knot_s[0];
    for (int i = 0; i + 1 < cf.f_n_knots; ++i)
        if (k <= cf.f_knot_step[i + 1]) return fmaf(cf.f_slope[i], (float)(k - cf.f_knot_step[i]), cf.f_knot_s[i]);
    return cf.f_knot_s[cf.f_n_knots - 1];
}

// h p and h at step k: the configuration's constants themselves without a
// schedule (the same bits as before schedules existed), else scaled by s(k)
__device__ __forceinline__ float field_hp(const DevCfg& cf, int64_t k)
{
    return cf.f_n_knots == 0 ? cf.hp : __fmul_rn(cf.hp, field_scale(cf, k));
}
__device__ __forceinline__ float field_h(const DevCfg& cf, int64_t k)
{
    return cf.f_n_knots == 0 ? cf.h : __fmul_rn(cf.h, field_scale(cf, k));
}

__device__ __forceinline__ StepConst step_const(const DevCfg& cf, float c)
{
    StepConst s;
    s.c = c;
    s.hdt = cf.hdt;
    s.dt = cf.dt;
    s.oma = cf.oma;
    s.inv1pa = cf.inv1pa;
    s.nqJx = cf.nqJx;
    s.nqJy = cf.nqJy;
    s.hp = cf.hp;
    s.q = cf.q;
    s.p = cf.p;
    return s;
}

// Coupling profiles of the anisotropic quench: J_par(k) = J_par a(k),
// J_perp(k) = J_perp b(k), piecewise linear through one knot grid and
// constant outside it, in FP32 like T(k); (1, 1) without a schedule.
__device__ __forceinline__ float2 coupling_scales(const DevCfg& cf, int64_t k)
{
    const int n = cf.c_n_knots;
    if (n <= 1 || k <= cf.c_knot_step[0])
        return n == 0 ? make_float2(1.f, 1.f) : make_float2(cf.c_knot_a[0], cf.c_knot_b[0]);
    for (int i = 0; i + 1 < n; ++i)
        if (k <= cf.c_knot_step[i + 1]) {
            const float dk = (float)(k - cf.c_knot_step[i]);
            return make_float2(fmaf(cf.c_slope_a[i], dk, cf.c_knot_a[i]), fmaf(cf.c_slope_b[i], dk, cf.c_knot_b[i]));
        }
    return make_float2(cf.c_knot_a[n - 1], cf.c_knot_b[n - 1]);
}

// J_par(k), J_perp(k): the configuration's own without a schedule (the same
// bits as before schedules existed), else scaled by the profiles
__device__ __forceinline__ float2 couplings_at(const DevCfg& cf, int64_t k)
{
    if (cf.c_n_knots == 0) return make_float2(cf.Jx, cf.Jy);
    const float2 ab = coupling_scales(cf, k);
    return make_float2(__fmul_rn(cf.Jx, ab.x), __fmul_rn(cf.Jy, ab.y));
}

// The constants of step k: noise amplitude c_k, the field's h_k p, and the
// couplings' -q J_par(k), -q J_perp(k).
__device__ __forceinline__ StepConst step_const_k(const DevCfg& cf, int64_t k, float c)
{
    StepConst s = step_const(cf, c);
    s.hp = field_hp(cf, k);
    if (cf.c_n_knots != 0) {
        const float2 ab = coupling_scales(cf, k);
        s.nqJx = __fmul_rn(cf.nqJx, ab.x);
        s.nqJy = __fmul_rn(cf.nqJy, ab.y);
    }
    return s;
}

// -------------------------------------------------------------------------
// One site of the merged BBK step (App. A.1) in leapfrog form.
// Stored state: theta_k and v_k = omega_{k-1/2}.  With g = (dt/2) F_k + c_k n_k:
//   omega_k     = (v_k + g) / (1 + eta dt / 2)          (end of Eq. BBK-2 of step k-1)
//   v_{k+1}     = (1 - eta dt / 2) omega_k + g           (Eq. BBK-1 of step k)
//   theta_{k+1} = wrap(theta_k + dt v_{k+1})             (drift + modulo)
// -------------------------------------------------------------------------

// Force on one site from its own (s, c) = (sin q t, cos q t), the sums of the
// neighbours' (s, c) along x and y, and sin(p t):
//   F = -q J_par (s (cL + cR) - c (sL + sR)) - q J_perp (s (cU + cD) - c (sU + sD)) + h p sin(p t)
__device__ __forceinline__ float site_force(const StepConst& K, float s, float c, float sx, float cx,
                                            float sy, float cy, float sinp)
{
    const float ax = fmaf(s, cx, -__fmul_rn(c, sx));
    const float ay = fmaf(s, cy, -__fmul_rn(c, sy));
    return fmaf(K.nqJx, ax, fmaf(K.nqJy, ay, __fmul_rn(K.hp, sinp)));
}

struct SiteOut {
    float theta, v, omega;
};

__device__ __forceinline__ SiteOut site_update(const StepConst& K, float theta, float v, float F, float cn)
{
    SiteOut o;
    const float g = fmaf(K.hdt, F, cn);
    o.omega = __fmul_rn(__fadd_rn(v, g), K.inv1pa);
    o.v = fmaf(K.oma, o.omega, g);
    o.theta = wrap_angle(fmaf(K.dt, o.v, theta));
    return o;
}

// The four sites of a quad at once: (s, c) = (sin q t, cos q t) of the quad,
// of its x neighbours (sL, cL left of site 0; sR, cR right of site 3) and of
// the quads above and below (P, N), v and the noise cn.  The same roundings as
// site_force and site_update.
struct QuadOut {
    P4 theta, v, omega;
};
__device__ __forceinline__ QuadOut quad_update(const StepConst& K, const P4& th, const P4& v, const P4& cn, const P4& s,
                                               const P4& c, float sL, float cL, float sR, float cR, const P4& Ps,
                                               const P4& Pc, const P4& Ns, const P4& Nc)
{
    // minus the sums of the neighbours' sines (scalar adds negate their operands
    // for free; a packed add would need a packed negation), the cosines' sums
    const P4 sx{make_float2(__fadd_rn(-sL, -s.a.y), __fadd_rn(-s.a.x, -s.b.x)),
                make_float2(__fadd_rn(-s.a.y, -s.b.y), __fadd_rn(-s.b.x, -sR))};
    const P4 sy{make_float2(__fadd_rn(-Ps.a.x, -Ns.a.x), __fadd_rn(-Ps.a.y, -Ns.a.y)),
                make_float2(__fadd_rn(-Ps.b.x, -Ns.b.x), __fadd_rn(-Ps.b.y, -Ns.b.y))};
    const P4 cx{make_float2(__fadd_rn(cL, c.a.y), __fadd_rn(c.a.x, c.b.x)),
                make_float2(__fadd_rn(c.a.y, c.b.y), __fadd_rn(c.b.x, cR))};
    const P4 cy = add4(Pc, Nc);
    const P4 ax = fma4(s, cx, mul4(c, sx)), ay = fma4(s, cy, mul4(c, sy));
    const P4 pt = mul4(K.p, th);
    const P4 sp{make_float2(__sinf(pt.a.x), __sinf(pt.a.y)), make_float2(__sinf(pt.b.x), __sinf(pt.b.y))};
    const P4 F = fma4(K.nqJx, ax, fma4(K.nqJy, ay, mul4(K.hp, sp)));
    const P4 g = fma4(K.hdt, F, cn);
    QuadOut o;
    o.omega = mul4(K.inv1pa, add4(v, g));
    o.v = fma4(K.oma, o.omega, g);
    o.theta = wrap_angle4(fma4(K.dt, o.v, th));
    return o;
}

// (sin q t, cos q t) of a quad
__device__ __forceinline__ void quad_sc(float q, const P4& th, P4& s, P4& c)
{
    const P4 a = mul4(q, th);
    __sincosf(a.a.x, &s.a.x, &c.a.x);
    __sincosf(a.a.y, &s.a.y, &c.a.y);
    __sincosf(a.b.x, &s.b.x, &c.b.x);
    __sincosf(a.b.y, &s.b.y, &c.b.y);
}

// Energy of one site with its forward bonds (x+1, y+1), per Eq. (XY-Hamilton-Kinetic),
// relative to the reference e_ref <= the potential part at every step:
//   omega^2 / 2 - J_par cos q(t - t_{x+1}) - J_perp cos q(t - t_{y+1}) + h cos(p t) - e_ref
// with cos q(a - b) = c_a c_b + s_a s_b, bx, by those bond cosines.  The
// potential terms are added to the small h cos(p t) - e_ref first, so every
// rounding is relative to the (small) result; the caller adds N e_ref back in FP64.
__device__ __forceinline__ float site_energy_rel(float omega, float bx, float by, float cosp, float Jx, float Jy,
                                                 float h, float e_ref)
{
    float e = fmaf(h, cosp, -e_ref);
    e = fmaf(-Jx, bx, e);
    e = fmaf(-Jy, by, e);
    return fmaf(__fmul_rn(0.5f, omega), omega, e);
}

// The four sites of a quad at once, with the same roundings: (s, c) of the quad, of
// the quad below (N) and of the site to its right (sR, cR).
__device__ __forceinline__ P4 quad_energy_rel(float p, float2 J, float h, float e_ref, const P4& s, const P4& c,
                                              const P4& Ns, const P4& Nc, float sR, float cR, const P4& om, const P4& th)
{
    const P4 sr{make_float2(s.a.y, s.b.x), make_float2(s.b.y, sR)}, cr{make_float2(c.a.y, c.b.x), make_float2(c.b.y, cR)};
    const P4 bx = fma4(c, cr, mul4(s, sr)), by = fma4(c, Nc, mul4(s, Ns));
    const P4 pt = mul4(p, th);
    const P4 cp{make_float2(__cosf(pt.a.x), __cosf(pt.a.y)), make_float2(__cosf(pt.b.x), __cosf(pt.b.y))};
    const P4 ref{splat2(-e_ref), splat2(-e_ref)};
    return fma4(mul4(0.5f, om), om, fma4(-J.y, by, fma4(-J.x, bx, fma4(h, cp, ref))));
}

// Jk: the couplings (couplings_at) and hk the field (field_h) of the recorded step
__device__ __forceinline__ float site_energy(const DevCfg& cf, float2 Jk, float hk, float omega, float s, float c,
                                             float sR, float cR, float sD, float cD, float cosp)
{
    const float bx = fmaf(c, cR, __fmul_rn(s, sR));
    const float by = fmaf(c, cD, __fmul_rn(s, sD));
    return site_energy_rel(omega, bx, by, cosp, Jk.x, Jk.y, hk, cf.e_ref);
}

// Asynchronous global -> shared copies (cp.async), issued by one lane for its
// own slot and read back by the same lane after cp_async_wait<N>() (this
// lane's groups but the newest N have landed): rows of the next iterations are
// in flight while the current one is computed, without a barrier.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Programmatic dependent launch: a kernel launched so (launch_dependent) may start
// while the launch before it on its stream drains.  dependency_wait() returns when
// that launch has completed and its writes are visible; what comes before it may
// read only what no launch of the same chunk of steps writes.  launch_next() lets
// the following launch start once every block has called it or ended.
// Every block of such a kernel calls dependency_wait(), also one that has nothing to
// do: what comes after a chain of launches waits for its last launch only, and that
// one completes after the others because each of its blocks has waited for the one
// before.  (A launch whose blocks all left without waiting could complete first.)
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ float4 ld4_stream(const float* p) { return __ldcs(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ void st4_stream(float* p, float4 v) { __stcs(reinterpret_cast<float4*>(p), v); }

__device__ __forceinline__ float f4get(const float4& v, int i)
{
    return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}

}  // namespace xy
