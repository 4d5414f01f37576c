// xy_adjoint_back.cu -- reverse sweep of the pathwise adjoint with the states
// of each checkpoint segment integrated backward in time inside the reverse
// kernel (App. A.1 run in reverse), instead of being recomputed forward and
// stored.
//
// The BBK step in leapfrog variables (theta_k, v_k = omega_{k-1/2}) with
// a = eta dt / 2 and g_k = (dt/2) F(theta_k) + c_k n_k,
//   omega_k = (v_k + g_k) / (1 + a),  v_{k+1} = (1 - a) omega_k + g_k,
//   theta_{k+1} = wrap(theta_k + dt v_{k+1}),
// is inverted site by site once the noise n_k is regenerated from its
// counter:
//   theta_k = wrap(theta_{k+1} - dt v_{k+1}),
//   omega_k = (v_{k+1} - g_k) / (1 - a),  v_k = (1 + a) omega_k - g_k,
// where g_k needs F(theta_k), i.e. the recovered angles of the four
// neighbours.  A launch for step k reads the state of step k + 1 and the
// adjoints of step k + 1, writes the state of step k and the adjoints of
// step k, and does the reverse of step k (phase A: site-local adjoint, phase
// B: Hessian stencil) exactly as the band reverse kernel of xy_adjoint.cu.
// Each segment starts from the exact checkpoint (or final state) at its end,
// so rounding of the inversion does not carry across segments.
//
// The |M_k| term of the objective needs sign(M_k), a sum over the whole
// lattice of the angles recovered in the same launch.  Its contribution
// w_M sign(M_k) sigma q cos(q theta_k) / N to the adjoint of theta_k enters
// nothing else of step k, so it is added by the next launch (step k - 1)
// when it reads that adjoint: every launch writes per-block partial sums of
// M_k into a two-slot ring, and the next one sums them in a fixed order,
// records M_k and applies the deferred term.
#include <type_traits>

#include "xy_device.cuh"

namespace xy {

namespace {

constexpr unsigned kFullB = 0xFFFFFFFFu;
constexpr int kMaxBackWarps = 16;  // Lx <= 2048
constexpr int kStages = 3;

__device__ __forceinline__ int wrapb(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// (through L2: another block may have written the row, in this launch)
__device__ __forceinline__ float4 ldcg4(const float* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }

__device__ __forceinline__ P4 sub4(const P4& x, const P4& y) { return fma4(-1.0f, y, x); }

// theta_k = wrap(theta_{k+1} - dt v_{k+1}): the drift of step k undone, with
// one explicit rounding so that every block recovering a row gets its bits
__device__ __forceinline__ P4 undrift(const P4& t1, const P4& v1, float dt) { return wrap_angle4(fma4(-dt, v1, t1)); }

__device__ __forceinline__ float warp_sumf_b(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFullB, v, o);
    return v;
}

// Shared memory of one warp: the rows in flight (by iteration % 3), and the ends
// of its lanes' quads for the lanes beside (by iteration % 3).
struct BackWarp {
    float4 th[kStages][32], v[kStages][32], tb[kStages][32], vb[kStages][32];
    float4 sc[3][32];           // (sin q t, cos q t) of the first and of the last site
    float4 fb[3][32], bx[3][32];  // F-bar, and the bond cosines to the column x + 1
    float4 th0[2][32];          // theta_k, for the lane's own next iteration (by iteration % 2)
    float4 tbp[2][32];          // adjoint of theta without the Hessian stencil, likewise
};

// (sin q t, cos q t) of a row of theta_k
struct RowK {
    P4 s, c;
};

}  // namespace

// WIDE: Lx > 128 (a block spans one band of Lx / 128 strips); OBS: k > k0;
// BACK: the state of step k is recovered from that of step k + 1 (every
// launch but the first, which reads the final state itself); SCHED: some
// configuration of the launch has a field or coupling schedule (without one
// the step's constants are the configuration's own and no knot is searched).  At 128
// registers an SM partition holds four warps (16 per SM).
//
// What bounds it: the issue slots that dependent instructions leave empty; a row
// moves 32 bytes per site, which the launch needs a third of its time for.  So the
// four sites of a lane go as packed pairs, the sums for the gradient too; the
// stencil of phase B is formed from fluxes, each bond's term once (up and down, a
// row's flux is kept for the next one); quads' ends cross lanes and warps through
// shared memory, where a row's results wait for the next one too (eight pointers
// and twelve more values in registers spilled); and the noise of the next row is
// formed beside phase B, whose chain is short of independent work.  Unrolled by
// three, without copies of the window, the loop outgrew the instruction cache and
// gained nothing.  64 lattices of 256 x 256, 8-row bands, four slices at once: 200 ->
// 136 instructions per site, 35.8 -> 26.8 us per step (half of the issue slots).
//
// SWEEP (observed backward steps only): one launch reverses the steps R.k down to
// R.k_last.  The blocks of a lattice are a thread-block cluster (eight at most) and
// meet at its barrier after every step, so a small lattice pays a barrier per step
// where a launch per step paid its start, its prologue and the drain of the one
// before (4 lattices of 64 x 64: 8.6 -> 6.5 us per
// step, 12 at the start).
template <bool WIDE, bool OBS, bool BACK, bool SCHED, bool SWEEP>
__global__ void __launch_bounds__(512, 1) adjoint_back_kernel(const DevCfg* cfgs, const BandTask* tasks, int H,
                                                              BackArgs R, PhiloxKeys keys)
{
    extern __shared__ BackWarp s_warps[];
    __shared__ double s_red[kGacc + 1][kMaxBackWarps];
    __shared__ float s_wm1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const BandTask task = tasks[blockIdx.x];
    const DevCfg& cf = cfgs[task.cfg];
    const int Lx = cf.Lx, Ly = cf.Ly;
    const int G = WIDE ? 32 : (Lx >> 2);
    const int groups = 32 / G;
    const int grp = lane / G, lg = lane - grp * G;
    const int per_block = WIDE ? 1 : n_warps * groups;  // bands per block
    const int band_raw = WIDE ? task.band0 : task.band0 + warp * groups + grp;
    // lane groups past the last band recompute the last band (so every shuffle
    // and barrier runs converged) and store nothing
    const bool active = band_raw < task.n_bands;
    const int band = active ? band_raw : task.n_bands - 1;
    const int x = (WIDE ? warp * 128 : 0) + 4 * lg;
    const int y0 = band * H;
    // warp and lane of the quads beside
    const int wL = WIDE && lane == 0 ? (warp + n_warps - 1) % n_warps : warp;
    const int wR = WIDE && lane == 31 ? (warp + 1) % n_warps : warp;
    const int lL = grp * G + (lg + G - 1) % G, lR = grp * G + (lg + 1) % G;
    const int64_t b = cf.b_first + task.rep;
    const int64_t lat_off = cf.offset + (int64_t)task.rep * cf.N + x;
    const int slot_j = task.band0 / per_block;  // this block's partial of M
    const int n_parts = (task.n_bands + per_block - 1) / per_block;
    const float invN = 1.0f / (float)cf.N, wE = R.wE;
    const uint32_t cfgrep = ((uint32_t)cf.noise_cfg << 16) | (uint32_t)(cf.rep0 + task.rep);
    double total = 0.0;  // this thread's gradient sum over the steps
    for (int64_t k = R.k;; --k) {
    // one pointer and the other arrays' distances from it, which stay kernel
    // parameters in a launch of one step: eight pointers would take sixteen registers
    const float* in = R.th_in;
    int64_t d_v_in = R.d_v_in, d_tb_in = R.d_tb_in, d_vb_in = R.d_vb_in, d_th_out = R.d_th_out, d_v_out = R.d_v_out,
            d_tb_out = R.d_tb_out, d_vb_out = R.d_vb_out;
    if (SWEEP) {
        const int par = (int)((R.k - k) & 1);  // the buffers alternate from the first step on
        if (k < R.k) {
            const int64_t m = k + 1 - R.k0;  // the state of step k + 1: a checkpoint, or the last step's output
            in = m < R.n && m % R.seg == 0 ? R.ck + 2 * R.T * (m / R.seg) : R.sbuf + 2 * R.T * (R.sb ^ par ^ 1);
            d_v_in = 4 * R.T;
        }
        auto dist = [&](const float* q) { return (int64_t)((const char*)q - (const char*)in); };
        const float* out = R.sbuf + 2 * R.T * (R.sb ^ par);
        d_th_out = dist(out);
        d_v_out = d_th_out + 4 * R.T;
        d_tb_in = dist(R.adjb + 2 * R.T * (R.acur ^ par));
        d_vb_in = d_tb_in + 4 * R.T;
        d_tb_out = dist(R.adjb + 2 * R.T * (R.acur ^ par ^ 1));
        d_vb_out = d_tb_out + 4 * R.T;
    }
    char* const base = (char*)(in + lat_off);
    auto at = [&](int64_t dist, int o) { return reinterpret_cast<float*>(base + dist + 4 * (int64_t)o); };
    const StepConst K = SCHED ? step_const_k(cf, k, noise_amp(cf, k)) : step_const(cf, noise_amp(cf, k));
    const float q2 = K.q * K.q, hp2 = K.hp * cf.p;
    auto noise = [&](int o) {
        return p4(gauss4_scaled(philox4x32_10_rk(noise_counter((uint32_t)(o + x) >> 2, cfgrep, k, 0u), keys), K.c));
    };
    P4 nz = noise(wrapb(y0 - 1, Ly) * Lx);
    if (!SWEEP || k == R.k) dependency_wait();  // the states, adjoints and partial sums of the launch before
    // M_{k+1} from the previous step's partials (fixed order), recorded by
    // the lattice's first block; its sign weights the deferred |M| term
    if (warp == 0) {
        float w = 0.f;
        if (BACK) {
            const double* mp = R.mpart + (b * 2 + ((k + 1) & 1)) * R.P;
            double m = 0.0;
            for (int j = lane; j < n_parts; j += 32) m += __ldcg(&mp[j]);
            for (int o = 1; o < 32 && o < n_parts; o <<= 1) m += __shfl_xor_sync(kFullB, m, o);
            if (slot_j == 0 && lane == 0) R.rec[b * R.rec_stride + (k + 1 - R.k0)].x = m;  // N M_{k+1}
            const float wq = R.wM * invN * K.q;
            w = m > 0.0 ? wq : (m < 0.0 ? -wq : 0.f);
        }
        if (lane == 0) s_wm1 = w;  // (lane 0 has the full sum at any number of parts)
    }
    // configuration constants in registers (the cp.async statements clobber
    // memory, which would otherwise reload them from the descriptor every row)
    const float2 Jk = SCHED ? couplings_at(cf, k) : make_float2(cf.Jx, cf.Jy);
    const float2 abk = SCHED ? coupling_scales(cf, k) : make_float2(1.f, 1.f);
    const float Jx = Jk.x, Jy = Jk.y, hF = SCHED ? field_h(cf, k) : cf.h;
    const float q2Jx = q2 * Jx, q2Jy = q2 * Jy;
    const bool stag = cf.stag != 0;
    const float wEn = wE * invN;
    const float inv_oma = 1.0f / K.oma, opa = 2.0f - K.oma;  // 1 / (1 - a), 1 + a
    // per-lane sums, two sites each (both halves added at the end)
    const float2 z2 = make_float2(0.f, 0.f);
    float2 aJx = z2, aJy = z2, ah = z2, abar = z2, cbar = z2, sw2 = z2, sbx = z2, sby = z2, scp = z2, pm = z2;
    auto dot = [&](float2& acc, const P4& u, const P4& w) { acc = __ffma2_rn(u.b, w.b, __ffma2_rn(u.a, w.a, acc)); };
    auto add = [&](float2& acc, const P4& u) { acc = __fadd2_rn(acc, __fadd2_rn(u.a, u.b)); };

    const int N = Lx * Ly;
    auto adv = [&](int r) { return r + Lx == N ? 0 : r + Lx; };
    BackWarp& me = s_warps[warp];
    // iteration i works on row t = y0 - 1 + i (phase A) and row t - 1 (phase B); its
    // stage holds theta_in of row t + 1, v_in of row t + 1 (BACK) or t, tb and vb
    // of row t
    int o_ld = wrapb(y0, Ly) * Lx, o_ldt = wrapb(y0 - 1, Ly) * Lx;  // rows t + 1 and t of the next issue
    const int n_it = H + 2;
    auto issue = [&](int ii, int slot) {
        if (ii < n_it) {
            cp_async16(&me.th[slot][lane], at(0, o_ld));
            cp_async16(&me.v[slot][lane], at(d_v_in, BACK ? o_ld : o_ldt));
            cp_async16(&me.tb[slot][lane], at(d_tb_in, o_ldt));
            cp_async16(&me.vb[slot][lane], at(d_vb_in, o_ldt));
            o_ldt = o_ld;
            o_ld = adv(o_ld);
        }
        cp_async_commit();
    };
    int o_a = o_ldt, o_b = 0;  // rows t and t - 1
    issue(0, 0);
    issue(1, 1);
    const float4* sc_l = &s_warps[wL].sc[0][lL];
    const float4* sc_r = &s_warps[wR].sc[0][lR];
    const float* fb_l = &s_warps[wL].fb[0][lL].w;  // the bond cosines lie 3 * 32 float4 further
    const float* fb_r = &s_warps[wR].fb[0][lR].x;
    RowK k0, k1, k2;
    P4 gy{z2, z2};  // flux between the rows t - 2 and t - 1
    P4 bym;         // bond cosines between the rows t - 1 and t
    {
        // rows t - 1 and t of the first iteration
        const int r_m1 = wrapb(y0 - 2, Ly) * Lx, r_0 = o_a;
        P4 t0;
        if (BACK) {
            const P4 t = undrift(p4(ldcg4(at(0, r_m1))), p4(ldcg4(at(d_v_in, r_m1))), K.dt);
            quad_sc(K.q, t, k1.s, k1.c);
            // theta_{k+1}, v_{k+1} of row t stay in the last iteration's stage
            me.th[2][lane] = ldcg4(at(0, r_0));
            me.v[2][lane] = ldcg4(at(d_v_in, r_0));
            t0 = undrift(p4(me.th[2][lane]), p4(me.v[2][lane]), K.dt);
        } else {
            quad_sc(K.q, p4(ldcg4(at(0, r_m1))), k1.s, k1.c);
            t0 = p4(ldcg4(at(0, r_0)));
        }
        quad_sc(K.q, t0, k2.s, k2.c);
        me.th0[1][lane] = f4(t0);
        me.sc[2][lane] = make_float4(k2.s.a.x, k2.c.a.x, k2.s.b.y, k2.c.b.y);
        bym = fma4(k1.c, k2.c, mul4(k1.s, k2.s));
        me.fb[2][lane] = me.bx[2][lane] = me.tbp[1][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();  // s_wm1, and the ends of the first row
    const float wM1 = s_wm1;
    // Ends published in iteration i are read in iteration i + 1, on the other side
    // of iteration i's barrier: those of (sin, cos) before iteration i + 1's, those
    // of F-bar after it.  Three slots, so that what iteration i + 3 writes was read
    // before the barrier of iteration i + 2.
    // (P, C, D: theta_k of the rows t - 1, t, t + 1)
    auto body = [&](int i, int slot, RowK& P, RowK& C, RowK& D) {
        const int prev = slot == 0 ? 2 : slot - 1;
        cp_async_wait<kStages - 2>();  // this lane's copies of iteration i have landed
        const bool own = active && i >= 1 && i <= H;  // row t is the band's: stored and summed
        const P4 in = p4(me.th[slot][lane]), vin = p4(me.v[slot][lane]);
        const int own_slot = i & 1;
        const P4 thC = p4(me.th0[own_slot ^ 1][lane]);
        {
            const P4 thD = BACK ? undrift(in, vin, K.dt) : in;
            me.th0[own_slot][lane] = f4(thD);
            quad_sc(K.q, thD, D.s, D.c);
        }
        me.sc[slot][lane] = make_float4(D.s.a.x, D.c.a.x, D.s.b.y, D.c.b.y);
        // ---------------- phase A on row t
        P4 tb = p4(me.tb[slot][lane]);
        const P4 vb = p4(me.vb[slot][lane]);
        const int yw = wrapb(y0 - 1 + i, Ly);
        const float sgn = stag && (yw & 1) ? -1.f : 1.f;  // of the quad's sites 0 and 2 (x is a multiple of 4)
        const float2 sg = make_float2(sgn, stag ? -sgn : sgn);
        if (BACK) {
            // deferred |M_{k+1}| term of the adjoint of theta_{k+1} (step
            // k + 1 > k0 is always observed)
            const P4 a = mul4(K.q, p4(me.th[prev][lane]));
            const float2 w = __fmul2_rn(splat2(wM1), sg);
            tb.a = __ffma2_rn(w, make_float2(__cosf(a.a.x), __cosf(a.a.y)), tb.a);
            tb.b = __ffma2_rn(w, make_float2(__cosf(a.b.x), __cosf(a.b.y)), tb.b);
        }
        const float2 l = *(reinterpret_cast<const float2*>(sc_l + prev * 32) + 1);
        const float2 r = *reinterpret_cast<const float2*>(sc_r + prev * 32);
        const P4 &s = C.s, &c = C.c;
        const P4 sx{make_float2(-l.x - s.a.y, -s.a.x - s.b.x), make_float2(-s.a.y - s.b.y, -s.b.x - r.x)};
        const P4 cx{make_float2(l.y + c.a.y, c.a.x + c.b.x), make_float2(c.a.y + c.b.y, c.b.x + r.y)};
        const P4 sy{make_float2(-P.s.a.x - D.s.a.x, -P.s.a.y - D.s.a.y), make_float2(-P.s.b.x - D.s.b.x, -P.s.b.y - D.s.b.y)};
        const P4 cy = add4(P.c, D.c);
        const P4 ax = fma4(s, cx, mul4(c, sx)), ay = fma4(s, cy, mul4(c, sy));
        const P4 pt = mul4(K.p, thC);
        P4 sp, cp;
        __sincosf(pt.a.x, &sp.a.x, &cp.a.x);
        __sincosf(pt.a.y, &sp.a.y, &cp.a.y);
        __sincosf(pt.b.x, &sp.b.x, &cp.b.x);
        __sincosf(pt.b.y, &sp.b.y, &cp.b.y);
        const P4 F = fma4(K.nqJx, ax, fma4(K.nqJy, ay, mul4(K.hp, sp)));
        const P4 g = fma4(K.hdt, F, nz);
        P4 om, vk;  // omega_k, v_k
        if (BACK) {
            const P4 ng = mul4(-1.0f, g);
            om = mul4(inv_oma, add4(p4(me.v[prev][lane]), ng));
            vk = fma4(opa, om, ng);
        } else {
            vk = vin;
            om = mul4(K.inv1pa, add4(vk, g));
        }
        issue(i + kStages - 1, prev);  // (the slot's theta_{k+1} and v_{k+1} have been read)
        const P4 byn = fma4(c, D.c, mul4(s, D.s));  // bond to row t + 1
        P4 bx;
        bx.a = make_float2(fmaf(c.a.x, c.a.y, s.a.x * s.a.y), fmaf(c.a.y, c.b.x, s.a.y * s.b.x));  // to column x + 1
        bx.b = make_float2(fmaf(c.b.x, c.b.y, s.b.x * s.b.y), fmaf(c.b.y, r.y, s.b.y * r.x));
        const P4 vbt = fma4(K.dt, tb, vb);
        P4 omb = mul4(K.oma, vbt), gb = vbt, vbk{z2, z2};
        if (OBS) {
            omb = fma4(wEn, om, omb);
            tb = fma4(-wEn, F, tb);
            vbk = mul4(K.inv1pa, omb);
            gb = add4(gb, vbk);
        }
        const P4 fb = mul4(K.hdt, gb);
        // the field's diagonal Hessian term of phase B, h p^2 cos(p t) F-bar, is site-local
        me.tbp[own_slot][lane] = f4(fma4(mul4(hp2, cp), fb, tb));
        me.fb[slot][lane] = f4(fb);
        me.bx[slot][lane] = f4(bx);
        if (own) {
            pm = __ffma2_rn(sg, __fadd2_rn(s.a, s.b), pm);
            if (OBS) {
                dot(sw2, om, om);
                add(sbx, bx);
                add(sby, byn);
                add(scp, cp);
            }
            dot(aJx, fb, ax);
            dot(aJy, fb, ay);
            dot(ah, fb, sp);
            // the damping's two places, -om vbt from 1 - a and -om vbk from 1 / (1 + a)
            // ((vk + g) / (1 + a)^2 is om / (1 + a)), in one sum
            dot(abar, om, gb);
            dot(cbar, gb, nz);
            st4(at(d_vb_out, o_a), f4(vbk));
            if (BACK) {
                st4(at(d_th_out, o_a), f4(thC));
                st4(at(d_v_out, o_a), f4(vk));
            }
        }
        if (WIDE) __syncthreads(); else __syncwarp();
        // ---------------- phase B on row t - 1 (F-bar of rows t - 2, t - 1, t), from
        // the fluxes bond * (difference of F-bar) across its four bonds
        const int o_n = adv(o_a);
        nz = noise(o_n);  // of row t + 1
        {
            const float fl = fb_l[prev * 128], bl = fb_l[(3 + prev) * 128], fr = fb_r[prev * 128];
            const P4 f = p4(me.fb[prev][lane]), bxf = p4(me.bx[prev][lane]);
            const float el = bl * (f.a.x - fl);
            const P4 e = mul4(bxf, P4{make_float2(f.a.y - f.a.x, f.b.x - f.a.y), make_float2(f.b.y - f.b.x, fr - f.b.y)});
            const P4 hx{make_float2(e.a.x - el, e.a.y - e.a.x), make_float2(e.b.x - e.a.y, e.b.y - e.b.x)};
            const P4 gn = mul4(bym, sub4(fb, f));
            const P4 out = fma4(q2Jx, hx, fma4(q2Jy, sub4(gn, gy), p4(me.tbp[own_slot ^ 1][lane])));
            gy = gn;
            if (active && i >= 2) st4(at(d_tb_out, o_b), f4(out));
        }
        bym = byn;
        o_b = o_a;
        o_a = o_n;
    };
    int slot = 0;  // i % 3
#pragma unroll 1
    for (int i = 0; i < n_it; ++i) {
        body(i, slot, k1, k2, k0);
        k1 = k2;
        k2 = k0;
        slot = slot == 2 ? 0 : slot + 1;
    }
    cp_async_wait<0>();
    if (!SWEEP || k == R.k_last) launch_next();
    // per-block accumulators: FP32 warp butterflies, the warps and the steps
    // combined in FP64 in a fixed order; the partial of M_k goes to the ring
    auto both = [](float2 v) { return v.x + v.y; };
    const float vals[kGacc + 1] = {
        fmaf(-K.q, both(aJx), -wEn * both(sbx)) * abk.x,                              // d/d J_par (J_par(k) = J_par a(k))
        fmaf(-K.q, both(aJy), -wEn * both(sby)) * abk.y,                              // d/d J_perp (J_perp b(k))
        fmaf(K.p, both(ah), wEn * both(scp)) * (SCHED ? field_scale(cf, k) : 1.f),  // d/d h (h_k = h s(k))
        -both(abar), 0.f, both(cbar),
        wEn * fmaf(0.5f, both(sw2), fmaf(-Jx, both(sbx), fmaf(-Jy, both(sby), hF * both(scp)))),  // w_E E / N
        both(pm),                                                                      // sum of sigma sin(q theta_k)
    };
#pragma unroll
    for (int i = 0; i < kGacc + 1; ++i) {
        const float w = warp_sumf_b(vals[i]);
        if (lane == 0) s_red[i][warp] = w;
    }
    __syncthreads();
    if (threadIdx.x < kGacc + 1) {
        double p4s[4] = {0.0, 0.0, 0.0, 0.0};  // (an FP64 addition takes dozens of cycles: four chains)
        for (int w2 = 0; w2 < n_warps; ++w2) p4s[w2 & 3] += s_red[threadIdx.x][w2];
        const double acc = (p4s[0] + p4s[1]) + (p4s[2] + p4s[3]);
        if (threadIdx.x == kGacc) R.mpart[(b * 2 + (k & 1)) * R.P + slot_j] = acc;
        total += acc;
    }
    if (!SWEEP || k == R.k_last) break;
    // every block of the lattice has written its rows and its partial of M_k
    // (released to the cluster by the arrival)
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    }
    if (threadIdx.x < kGacc) R.gacc[(int64_t)(R.block_base + blockIdx.x) * kGacc + threadIdx.x] += total;
}

// Blocks of a lattice that one launch may sweep over its steps: the cluster size, or
// 0 where they are too many for a (portable) cluster.
int back_sweep_cluster(int blocks_per_lattice) { return blocks_per_lattice <= 8 ? blocks_per_lattice : 0; }

// sweep > 0: steps R.k .. R.k_last in one launch, clusters of `sweep` blocks (a
// lattice's blocks, consecutive tasks); 0: step R.k.
cudaError_t launch_adjoint_back(const DevCfg* d_cfg, const BandTask* tasks, int n_tasks, int Lx, int H, uint64_t seed,
                                bool back, int sweep, BackArgs R, bool after, cudaStream_t st)
{
    if (n_tasks == 0) return cudaSuccess;
    const bool wide = Lx > 128;
    const int threads = wide ? (Lx / 128) * 32 : 256;
    const int smem = (threads / 32) * (int)sizeof(BackWarp);
    const bool obs = R.k > R.k0;
    using Kern = void (*)(const DevCfg*, const BandTask*, int, BackArgs, PhiloxKeys);
#define BACK_ROW(W, S)                                                                                       \
    {{adjoint_back_kernel<W, false, false, S, false>, adjoint_back_kernel<W, false, true, S, false>},        \
     {adjoint_back_kernel<W, true, false, S, false>, adjoint_back_kernel<W, true, true, S, false>}}
    static const Kern table[2][2][2][2] = {{BACK_ROW(false, false), BACK_ROW(true, false)},
                                           {BACK_ROW(false, true), BACK_ROW(true, true)}};
#undef BACK_ROW
    static const Kern sweeps[2][2] = {
        {adjoint_back_kernel<false, true, true, false, true>, adjoint_back_kernel<true, true, true, false, true>},
        {adjoint_back_kernel<false, true, true, true, true>, adjoint_back_kernel<true, true, true, true, true>}};
    if (sweep > 0 && (!back || R.k_last <= R.k0 || n_tasks % sweep != 0)) return cudaErrorInvalidValue;
    const Kern kern = sweep > 0 ? sweeps[R.sched != 0][wide] : table[R.sched != 0][wide][obs][back];
    if (smem > 46 * 1024) {  // (the limit belongs to the kernel, which other shapes share: always the largest)
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   kMaxBackWarps * (int)sizeof(BackWarp));
        if (e != cudaSuccess) return e;
    }
    auto dist = [&](const float* q) { return q ? (int64_t)((const char*)q - (const char*)R.th_in) : 0; };
    R.d_v_in = dist(R.v_in);
    R.d_tb_in = dist(R.tb_in);
    R.d_vb_in = dist(R.vb_in);
    R.d_th_out = dist(R.th_out);
    R.d_v_out = dist(R.v_out);
    R.d_tb_out = dist(R.tb_out);
    R.d_vb_out = dist(R.vb_out);
    return launch_dependent(kern, (unsigned)n_tasks, (unsigned)threads, (size_t)smem, st, after, sweep, d_cfg, tasks, H, R,
                            philox_round_keys(seed));
}

}  // namespace xy
