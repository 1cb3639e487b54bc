// line_table.cuh -- the folded line sums of a model without a channel loop
// per spaxel.
//
// The line width is one number per model (Sec. 2.1.4), so the moment sums
// (q0, q1, q2) of a spaxel's line (fused_line.cuh, per unit amplitude) depend
// on the spaxel through its line-of-sight velocity v alone.  Two forms take
// the place of the 20 - 70 sampled channels:
//
//  * Lines whose window lies among the interior channels (those with the
//    whole LSF inside the band): the sums run over an unbroken row of
//    channels, and the Poisson summation formula gives them in closed form,
//      sum_e g(v_e - v)           = S (1 + 2 q cos t + 2 q^4 cos 2t)
//      sum_e g(v_e - v)(v_e - v)  = -S k (2 q sin t + 4 q^4 sin 2t)
//      sum_e g(v_e - v)(v_e - v)^2 = S (s^2 (1 + ..) - k^2 (2 q cos t + 8 q^4 cos 2t))
//    with g the Gaussian of width s, S = s sqrt(2 pi) / dv, k = 2 pi s^2 / dv,
//    q = exp(-2 pi^2 s^2 / dv^2), t = 2 pi (v - v_0) / dv.  For lines wider
//    than kLcSmooth channels the terms in q vanish in FP32; the next one,
//    q^9, is below 1e-9 down to kLcNarrow channels.
//  * Lines that reach the band edges: the velocities the model can reach are
//    cut into segments of at most kLtWidth line widths, aligned to the first
//    and last data channel (where the centre the sums are taken about is
//    clamped and their derivative jumps); each segment carries the degree-7
//    polynomials through the sums at its eight Chebyshev nodes, sampled
//    channel by channel once per CTA.
//
// Accuracy: the sums are sums of Gaussians of the line width, so the
// interpolation error of a 0.7 s segment is below 1e-8 of the sums' values
// inside the band and below 2e-7 up to kLtReach widths outside it (relative
// to the local, already truncated values), at and under the FP32 rounding of
// the sampled sums; lines as narrow as kLtNarrow channels included.  Lines
// further outside, narrower ones, models that would need more than kLtMaxSeg
// segments (a velocity range of many line widths, whose direct sum has few
// channels in its window) and images too small to pay for the nodes keep the
// direct sum (line_sums).
//
// Cost per spaxel beside the geometry: a few FMAs, or six 16-byte
// shared-memory loads (neighbouring spaxels mostly share a segment:
// broadcasts) and 21 FMAs, against about 9 instructions per channel pair.
#pragma once

#include "fused_line.cuh"

namespace gbk {

constexpr int kLtNodes = 8;             // nodes (and coefficients) per segment
constexpr int kLtMaxSeg = 64;
constexpr int kLtSegF = 3 * kLtNodes;   // floats per segment
constexpr int kLtLanes = 8;             // threads that share a node's channel sum
constexpr float kLtWidth = 0.7f;        // widest segment, in line widths
constexpr float kLtReach = 3.0f;        // line widths served beyond the data band
constexpr float kLtNarrow = 0.25f;      // narrowest line served by polynomials, in channels
constexpr float kLcNarrow = 0.45f;      // narrowest line served in closed form, in channels
constexpr float kLcSmooth = 1.15f;      // from here on the closed form has no ripple: 2 q = 9e-12
constexpr float kLcWindow = 6.0f;       // a line's half window for the closed form: the two
                                        // tails beyond hold 2e-9 of q0 and 7.5e-8 of q2

struct LineTab {
    int nseg;            // polynomial segments stored (0: none)
    int first, nb;       // index of the first segment reached (0 starts at v_lo), segments inside the band
    int int0, int1;      // segments [int0, int1) are served in closed form and not stored
    float w, inv_w, v0;  // segment width (km/s), start of the first segment reached
    float c0, c1;        // velocities of the closed form (empty: c0 > c1)
    float S, SV;         // S and S (s^2 + LSF variance)
    float h1, h4;        // 2 q, 2 q^4 (0 for smooth lines)
    float k, k2, s2v;    // 2 pi s^2 / dv, its square, s^2 + LSF variance
    float inv_dv;
};

// 1 / the unit of length of los_disc2: r_t held to [1e-12, 1e9] pixels.
// Below, atan(r / r_t) is pi/2 at every FP32 position but the centre itself;
// above, atan(u) / u is 1 and disc_const's k carries the rest.
__device__ __forceinline__ float disc_inv_unit(const ModelConst &c) { return fminf(fmaxf(c.inv_rt, 1e-9f), 1e12f); }

// The forms that serve a model (the same whatever the tiling, so are the
// sums).  A few dozen operations: one thread computes it for its block.
__device__ inline LineTab line_table_plan(const Geom &g, const ModelConst &c, const LineCtx &L)
{
    LineTab T = {};
    T.w = T.inv_w = 1.f;
    T.c0 = 1.f;
    T.c1 = -1.f;
    const float s = c.sigma;
    if (!c.valid || !(s >= kLtNarrow * g.dv)) return T;
    // los_disc2 squares lengths in units of r_t: where the farthest deprojected
    // one might overflow (r_t = 1e-12 px under more than 89.999 degrees, a
    // centre far outside the image) every spaxel takes the direct sum, whose
    // lengths are in pixels.
    const float far = (float)(g.ex + g.ey) + fabsf(c.x0) + fabsf(c.y0);
    if (!(far * c.inv_cos_i * disc_inv_unit(c) < 1e18f)) return T;
    const float B = L.v_hi - L.v_lo;
    if (B > 0.f) {
        const float nb = ceilf(B / (kLtWidth * s));
        if (!(nb <= 4096.f)) return T;
        T.nb = (int)nb;
        T.w = B / nb;
    } else {
        T.w = kLtWidth * s;
    }
    T.inv_w = 1.f / T.w;
    // |v_los - Vsys| < Vmax sin i (Eqs. 6 and 8)
    const float vm = fabsf(c.vrot_k * c.sin_i) * 1.5709f;
    const float lo = fmaxf(c.vsys - vm, L.v_lo - kLtReach * s);
    const float hi = fminf(c.vsys + vm, L.v_hi + kLtReach * s);
    const float f0 = floorf((lo - L.v_lo) * T.inv_w), f1 = floorf((hi - L.v_lo) * T.inv_w) + 1.f;
    if (!(f1 > f0)) return T;
    // the whole segments among the velocities that the closed form serves
    float i0 = f1, i1 = f1;
    if (s >= kLcNarrow * g.dv) {
        const float a = fmaf((float)L.elo, g.dv, L.vz0) + kLcWindow * s;
        const float b = fmaf((float)(L.ehi - 1), g.dv, L.vz0) - kLcWindow * s;
        const float j0 = fmaxf(ceilf((a - L.v_lo) * T.inv_w), f0), j1 = fminf(floorf((b - L.v_lo) * T.inv_w), f1);
        if (j1 > j0) {
            i0 = j0;
            i1 = j1;
            // a hair inside, so that a velocity that rounds out of these
            // segments is not taken for one in them
            T.c0 = fmaf(j0 + 1e-4f, T.w, L.v_lo);
            T.c1 = fmaf(j1 - 1e-4f, T.w, L.v_lo);
            T.inv_dv = 1.f / g.dv;
            T.S = s * 2.5066282746310002f * T.inv_dv;
            T.s2v = fmaf(s, s, L.var_z);
            T.SV = T.S * T.s2v;
            const float r = s * T.inv_dv;
            if (r < kLcSmooth) {
                const float x = 19.739208802178716f * r * r;  // 2 pi^2 s^2 / dv^2
                T.h1 = 2.f * expf(-x);
                T.h4 = 2.f * expf(-4.f * x);
                T.k = 6.283185307179586f * s * r;
                T.k2 = T.k * T.k;
            }
        }
    }
    T.first = (int)f0;
    T.int0 = (int)i0;
    T.int1 = (int)i1;
    T.v0 = fmaf(f0, T.w, L.v_lo);
    const float n = (f1 - f0) - (i1 - i0);
    if (n <= (float)kLtMaxSeg && 2.f * kLtNodes * n <= (float)g.ex * (float)g.ey) T.nseg = (int)n;
    return T;
}

// Builds the polynomials of T in tab[kLtSegF * T.nseg] (shared memory) with
// all `nthr` (a multiple of 32) threads of the block; ends with a barrier.
// `edge` holds the three edge tables of etl floats each.
__device__ inline void line_table_build(const Geom &g, const LineCtx &L, const LineTab &T, const float *edge, int etl,
                                        float *tab, int tid, int nthr)
{
    const float *const eG0 = edge, *const eA1 = edge + etl, *const eA2 = edge + 2 * etl;
    // cos((2 i + 1) pi / 16)
    const float X[4] = {0.98078528f, 0.83146961f, 0.55557023f, 0.19509032f};
    const int sub = tid & (kLtLanes - 1);
    const int nodes = kLtNodes * T.nseg;
    const float ref_lo = fmaf(L.eref_lo, g.dv, L.vz0), ref_hi = fmaf(L.eref_hi, g.dv, L.vz0);
    for (int n0 = 0; n0 < nodes; n0 += nthr / kLtLanes) {  // whole warps
        const int node = n0 + tid / kLtLanes;
        const int i = node & (kLtNodes - 1);
        int seg = T.first + node / kLtNodes;
        if (seg >= T.int0) seg += T.int1 - T.int0;
        const int j = i < 4 ? i : 7 - i;
        const float xa = (j & 2) ? ((j & 1) ? X[3] : X[2]) : ((j & 1) ? X[1] : X[0]);
        const float xi = i < 4 ? -xa : xa;
        const float v = fmaf((float)seg + 0.5f + 0.5f * xi, T.w, L.v_lo);
        const float a = seg < 0 ? L.v_lo : (seg >= T.nb ? L.v_hi : v);
        const float sh = v - a;
        const float ub = L.al * (L.vz0 - v);  // u = alpha (v_e - v) at e = 0
        const float cut = kUCut + L.al * fabsf(sh);
        const int e0 = max(0, (int)floorf((-cut - ub) * L.inv_adv));
        const int e1 = node < nodes ? min(g.ez, (int)ceilf((cut - ub) * L.inv_adv) + 1) : 0;
        // interior channels take the offset from the Gaussian's own argument,
        // so that a symmetric line's first moment cancels
        float q0 = 0.f, q1 = 0.f, q2 = 0.f;
        for (int e = e0 + sub; e < e1; e += kLtLanes) {
            const float u = fmaf((float)e, L.adv, ub);
            const float gs = ex2_approx(-u * u);
            float G = 1.f, b1 = 0.f, b2 = L.var_z, d = fmaf(u, L.inv_al, sh);
            if (e < L.elo || e >= L.ehi) {
                const int slot = e < L.elo ? e : L.hi_off + (e - L.ehi);
                G = eG0[slot];
                b1 = eA1[slot];
                b2 = eA2[slot];
                d = (e < L.elo ? ref_lo : ref_hi) - a;
            }
            q0 = fmaf(gs, G, q0);
            q1 = fmaf(gs, fmaf(d, G, b1), q1);
            q2 = fmaf(gs, fmaf(d, fmaf(d, G, b1 + b1), b2), q2);
        }
#pragma unroll
        for (int off = kLtLanes / 2; off > 0; off >>= 1) {
            q0 += __shfl_xor_sync(0xffffffffu, q0, off);
            q1 += __shfl_xor_sync(0xffffffffu, q1, off);
            q2 += __shfl_xor_sync(0xffffffffu, q2, off);
        }
        if (node < nodes && sub == 0) {
            float *o = tab + (node / kLtNodes) * kLtSegF + 3 * i;
            o[0] = q0;
            o[1] = q1;
            o[2] = q2;
        }
    }
    __syncthreads();
    // Node values f_i to monomial coefficients in t in [-1, 1], in place, one
    // thread per segment and sum: Chebyshev coefficients by the discrete
    // cosine sums of the even and odd parts of f_i - f_4 (the differences are
    // near exact, so a constant keeps its rounding), then powers of t.  Going
    // through the rapidly falling Chebyshev coefficients keeps the large
    // factors of the high powers off the rounding of the node values.
    for (int k = tid; k < 3 * T.nseg; k += nthr) {
        float *o = tab + (k / 3) * kLtSegF + k % 3;
        float f[kLtNodes];
#pragma unroll
        for (int i = 0; i < kLtNodes; ++i) f[i] = o[3 * i];
        const float base = f[4];
        float ev[4], od[4];  // nodes -X[i] (f[i]) and +X[i] (f[7 - i])
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float p = f[7 - i] - base, m = f[i] - base;
            ev[i] = 0.25f * (p + m);
            od[i] = 0.25f * (p - m);
        }
        // c_k = (2/8) sum_i f_i cos(k (2 i + 1) pi / 16)
        const float c2 = 0.92387953f, s2 = 0.38268343f, r2 = 0.70710678f;
        const float C0 = 0.5f * ((ev[0] + ev[3]) + (ev[1] + ev[2]));
        const float C2 = c2 * (ev[0] - ev[3]) + s2 * (ev[1] - ev[2]);
        const float C4 = r2 * ((ev[0] + ev[3]) - (ev[1] + ev[2]));
        const float C6 = s2 * (ev[0] - ev[3]) - c2 * (ev[1] - ev[2]);
        const float C1 = X[0] * od[0] + X[1] * od[1] + X[2] * od[2] + X[3] * od[3];
        const float C3 = X[1] * od[0] - X[3] * od[1] - X[0] * od[2] - X[2] * od[3];
        const float C5 = X[2] * od[0] - X[0] * od[1] + X[3] * od[2] + X[1] * od[3];
        const float C7 = X[3] * od[0] - X[2] * od[1] + X[1] * od[2] - X[0] * od[3];
        o[0] = base + (C0 - C2 + C4 - C6);
        o[3] = C1 - 3.f * C3 + 5.f * C5 - 7.f * C7;
        o[6] = 2.f * C2 - 8.f * C4 + 18.f * C6;
        o[9] = 4.f * C3 - 20.f * C5 + 56.f * C7;
        o[12] = 8.f * C4 - 48.f * C6;
        o[15] = 16.f * C5 - 112.f * C7;
        o[18] = 32.f * C6;
        o[21] = 64.f * C7;
    }
    __syncthreads();
}

// Neither form serves any of the model's lines.
__device__ __forceinline__ bool line_table_empty(const LineTab &T) { return T.nseg == 0 && T.c0 > T.c1; }

// The polynomials' sums (q0, q1, q2) at position t of a stored segment.
__device__ __forceinline__ void line_table_eval(const float *tab, int seg, float t, float &q0, float &q1, float &q2)
{
    const float4 *p = reinterpret_cast<const float4 *>(tab + seg * kLtSegF);
    float f[kLtSegF];
#pragma unroll
    for (int i = 0; i < kLtSegF / 4; ++i) {
        const float4 v = p[i];
        f[4 * i] = v.x; f[4 * i + 1] = v.y; f[4 * i + 2] = v.z; f[4 * i + 3] = v.w;
    }
    q0 = f[21]; q1 = f[22]; q2 = f[23];
#pragma unroll
    for (int k = kLtNodes - 2; k >= 0; --k) {
        q0 = fmaf(q0, t, f[3 * k]);
        q1 = fmaf(q1, t, f[3 * k + 1]);
        q2 = fmaf(q2, t, f[3 * k + 2]);
    }
}

// The closed form at velocity v; vz0: velocity of extended channel 0.
__device__ __forceinline__ void line_closed(const LineTab &T, float vz0, float v, float &q0, float &q1, float &q2)
{
    q0 = T.S;
    q1 = 0.f;
    q2 = T.SV;
    if (T.h1 != 0.f) {  // uniform over the model
        const float x = (v - vz0) * T.inv_dv;
        // 2 pi times the phase in [-1/2, 1/2]; sin and cos to about 1e-6,
        // times 2 q <= 0.04
        const float ph = 6.283185307179586f * (x - rintf(x));
        const float sn = __sinf(ph), cs = __cosf(ph);
        const float a = T.h1 * cs, b = T.h4 * fmaf(2.f * cs, cs, -1.f);  // 2 q cos t, 2 q^4 cos 2t
        q0 = T.S * (1.f + (a + b));
        q1 = -T.S * T.k * sn * fmaf(4.f * T.h4, cs, T.h1);
        q2 = T.S * fmaf(-T.k2, fmaf(4.f, b, a), T.s2v * (1.f + (a + b)));
    }
}

// Line-of-sight velocity (Eq. 8) and the line amplitude times the surface
// brightness (Eq. 5, per unit I0) at sky positions (x, y) and (x, y + 1), two
// rows in the lanes of f32x2 operations.  Lengths are in units of r_t, so
// with u = r / r_t the velocity is Vsys + (2/pi) Vmax sin i (x_e / r_t)
// atan(u) / u: atan(s) / s is a polynomial in s^2 on [0, 1] (minimax in
// relative error found by a Remez exchange; 5e-9 with its constants rounded
// to FP32), taken at s = u, or at
// s = 1/u with atan(u) = pi/2 - atan(1/u); both u and 1/u come from one
// reciprocal square root, and no division is left.  One Newton step refines
// both: over 46 cases of the declared ranges the velocity maps' error against
// 64 bits is then 1.01 times that of a square root and a division, 1.02 times
// with 1/u as the instruction gives it; the step's time does not show.
struct DiscConst {
    float x0, y0, a1, a2, b1, b2;  // x_e / r_t = a1 dx + a2 dy, -y_e / (r_t cos i) = b1 dx + b2 dy
    float vsys, k, hl, A;
};

__device__ __forceinline__ f32x2 dup2(float v) { return pk2(v, v); }

__device__ __forceinline__ DiscConst disc_const(const ModelConst &c)
{
    const float ir = disc_inv_unit(c);
    DiscConst d;
    d.x0 = c.x0;
    d.y0 = c.y0;
    d.a1 = -c.sin_pa * ir;
    d.a2 = c.cos_pa * ir;
    d.b1 = c.cos_pa * c.inv_cos_i * ir;
    d.b2 = c.sin_pa * c.inv_cos_i * ir;
    d.vsys = c.vsys;
    d.k = c.vrot_k * c.sin_i * fminf(1.f, c.inv_rt * 1e9f);
    d.hl = -1.4426950408889634f * c.inv_h / ir;
    d.A = c.amp;
    return d;
}

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// atan(s) / s for 0 <= s <= 1 (scalar: its constants ride in the FMAs, packed
// they would each take a register pair).
__device__ __forceinline__ float atan_over(float s)
{
    const float z = s * s;
    float p = -1.7539301e-3f;
    p = fmaf(p, z, 1.0726944e-2f);
    p = fmaf(p, z, -3.0804597e-2f);
    p = fmaf(p, z, 5.7552103e-2f);
    p = fmaf(p, z, -8.3773158e-2f);
    p = fmaf(p, z, 1.0942031e-1f);
    p = fmaf(p, z, -1.4261933e-1f);
    p = fmaf(p, z, 1.9998266e-1f);
    p = fmaf(p, z, -3.3333284e-1f);
    return fmaf(p, z, 1.f);
}

__device__ __forceinline__ void los_disc2(const DiscConst &d, float x, float y, float &v0, float &v1, float &A0,
                                          float &A1)
{
    const float dx = x - d.x0, dya = y - d.y0, dyb = (y + 1.f) - d.y0;
    const float xa = dx * d.a1, ya = dx * d.b1;
    const f32x2 xe = pk2(fmaf(dya, d.a2, xa), fmaf(dyb, d.a2, xa));      // Eq. 1
    const f32x2 yd = pk2(fmaf(dya, d.b2, ya), fmaf(dyb, d.b2, ya));      // -Eq. 2, deprojected
    float wa, wb, ua, ub, ta, tb;
    upk2(fma2(xe, xe, mul2(yd, yd)), wa, wb);                            // u^2 (Eq. 3)
    wa = fmaxf(wa, 1e-36f);
    wb = fmaxf(wb, 1e-36f);
    ta = rsqrt_approx(wa);
    tb = rsqrt_approx(wb);
    const f32x2 t = pk2(ta, tb), u0 = mul2(pk2(wa, wb), t);
    const f32x2 nt = fma2(mul2(u0, t), dup2(-0.5f), dup2(1.5f));         // one Newton step
    const f32x2 u = mul2(u0, nt);
    upk2(mul2(t, nt), ta, tb);                                           // 1 / u
    upk2(u, ua, ub);
    const float pa = atan_over(fminf(ua, ta)), pb = atan_over(fminf(ub, tb));
    float fa, fb;
    fa = ua > 1.f ? fmaf(-ta, pa, 1.57079633f) * ta : pa;                // atan(u) / u
    fb = ub > 1.f ? fmaf(-tb, pb, 1.57079633f) * tb : pb;
    upk2(mul2(xe, pk2(fa, fb)), fa, fb);
    v0 = fmaf(d.k, fa, d.vsys);                                          // Eq. 8
    v1 = fmaf(d.k, fb, d.vsys);
    A0 = d.A * ex2_approx(d.hl * ua);                                    // Eq. 5
    A1 = d.A * ex2_approx(d.hl * ub);
}

// The line sums of a spaxel with velocity v that the closed form does not
// serve (per unit amplitude); NaN in q.x, and `left` set, where the polynomials
// do not either.
__device__ __forceinline__ float4 line_sums_edge(const LineCtx &L, const LineTab &T, const float *tab, float v,
                                                 bool &left)
{
    float4 q;
    const float p = (v - T.v0) * T.inv_w, fl = floorf(p);
    const int seg = (int)fl, lows = T.int0 - T.first, gap = T.int1 - T.int0;
    // a velocity just inside the closed form's outermost segments belongs to
    // the stored neighbour, whose polynomial reaches that far
    int st;
    float t = fmaf(2.f, p - fl, -1.f);
    if (seg < lows) {
        st = seg;
    } else if (seg >= lows + gap) {
        st = seg - gap;
    } else if (2.f * (p - (float)lows) < (float)gap) {
        st = lows - 1;
        t += 2.f * (float)(seg - st);
    } else {
        st = lows;
        t -= 2.f * (float)(lows + gap - seg);
    }
    if (p >= 0.f && st >= 0 && st < T.nseg) {
        line_table_eval(tab, st, t, q.x, q.y, q.z);
    } else {
        q.x = q.y = q.z = __int_as_float(0x7fc00000);
        left = true;
    }
    q.w = fminf(fmaxf(v, L.v_lo), L.v_hi);
    return q;
}

// The line sums (A q0, A q1, A q2, a) of the spaxels at (x, y) and (x, y + 1),
// per unit I0; NaN in q[h].x, and `left` set, where only the direct sum serves.
__device__ __forceinline__ void line_sums_pair(const DiscConst &d, const LineCtx &L, const LineTab &T,
                                               const float *tab, float x, float y, float4 (&q)[2], bool &left)
{
    float v[2], A[2];
    los_disc2(d, x, y, v[0], v[1], A[0], A[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (v[h] >= T.c0 && v[h] <= T.c1) {
            line_closed(T, L.vz0, v[h], q[h].x, q[h].y, q[h].z);
            q[h].w = v[h];
        } else {
            q[h] = line_sums_edge(L, T, tab, v[h], left);
        }
        q[h].x *= A[h];
        q[h].y *= A[h];
        q[h].z *= A[h];
    }
}

}  // namespace gbk
