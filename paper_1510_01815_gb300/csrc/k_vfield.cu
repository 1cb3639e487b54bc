// k_vfield.cu -- the velocity-field modelling strategy (Sec. 2.2.1): Eq. 8
// evaluated at every data pixel directly, with the arctan (Eq. 6) or the
// Epinat (Eq. 7) rotation curve, then the residuals and chi-squared of
// Eq. 11.  There is no cube and no PSF or LSF; m0 = 1 (every pixel valid)
// and m2 = sigma0, the constant dispersion model of Sec. 2.1.4.
//
// The sums have a fixed order, so chi2 and the normal matrix are bitwise
// reproducible: 256 chains per model, chain t taking pixels t, t + 256, ..
// in turn, FP32 sums over each 32 chains and FP64 over the eight groups.  A
// chain is serial but its terms are not: where the models do not fill the chip
// a model has a cluster of eight CTAs, one per group of 32 chains, and the
// eight warps of a CTA evaluate eight consecutive steps of its chains at once,
// hand the terms over in shared memory (double-buffered, one barrier per eight
// steps) and add them up in the chains' order, each warp its share of the
// entries.  Batches that fill the chip take one CTA per model and one thread
// per chain.  64 Epinat fields of 256 x 256: chi2 229 us with a CTA each (64
// SMs, two warps a scheduler, a chain of powers and divisions 256 pixels
// long), 60 us with a cluster each; the normal equations 279 and 139 us.  1024
// of them: 549 and 1308 us with a CTA each, 678 and 1553 us with a cluster.
// The powers, logarithms and divisions (about 250 instructions a pixel) bound
// both.
#include <cooperative_groups.h>

#include <algorithm>

#include "gbk_api_internal.h"
#include "k_fused.h"
#include "k_tangent.h"

namespace cg = cooperative_groups;

namespace gbk {

constexpr int kVfThreads = 256;

struct VfConst {
    float x0, y0, sin_pa, cos_pa, sin_i, inv_cos_i, vsys, sig0;
    float vk, inv_rt;   // arctan: (2/pi) Vmax and 1/r_t; Epinat: V_t and 1/r_t
    float a, g;         // Epinat slopes
    int epinat, valid;
};

__device__ inline VfConst vf_const(const double *p, int model)
{
    VfConst c;
    c.epinat = model == GBK_MODEL_VFIELD_EPINAT;
    bool ok = (p[GBK_INCL] >= 0.0) && (p[GBK_INCL] < 90.0) && (p[GBK_RT] > 0.0) && (p[GBK_SIG0] >= 0.0);
    for (int k = 0; k <= GBK_SIG0; ++k) ok = ok && isfinite(p[k]);
    if (c.epinat) ok = ok && isfinite(p[GBK_EPI_A]) && isfinite(p[GBK_EPI_G]);
    c.valid = ok ? 1 : 0;
    float sp, cp, si, ci;
    sincospif((float)(p[GBK_PA] * (1.0 / 180.0)), &sp, &cp);
    sincospif((float)(p[GBK_INCL] * (1.0 / 180.0)), &si, &ci);
    c.x0 = (float)p[GBK_X0];
    c.y0 = (float)p[GBK_Y0];
    c.sin_pa = sp;
    c.cos_pa = cp;
    c.sin_i = si;
    c.inv_cos_i = 1.0f / ci;
    c.vsys = (float)p[GBK_VSYS];
    c.sig0 = (float)p[GBK_SIG0];
    c.vk = c.epinat ? (float)p[GBK_VMAX] : (float)(0.63661977236758134 * p[GBK_VMAX]);
    c.inv_rt = 1.0f / (float)p[GBK_RT];
    c.a = c.epinat ? (float)p[GBK_EPI_A] : 0.f;
    c.g = c.epinat ? (float)p[GBK_EPI_G] : 0.f;
    return c;
}

// Eq. 8 at pixel (x, y): Vsys + [Vrot(r)/r] x_e sin i (Eqs. 1-4, 6 or 7).
__device__ __forceinline__ float vf_velocity(const VfConst &c, float x, float y)
{
    float dx = x - c.x0, dy = y - c.y0;
    float xe = -dx * c.sin_pa + dy * c.cos_pa;  // Eq. 1
    float ye = -dx * c.cos_pa - dy * c.sin_pa;  // Eq. 2
    float yd = ye * c.inv_cos_i;
    float r = sqrtf(xe * xe + yd * yd);         // Eq. 3
    float f;
    if (c.epinat) {
        float q = r * c.inv_rt;
        f = (r > 0.f) ? c.vk * powf(q, c.g) / ((1.f + powf(q, c.a)) * r) : 0.f;  // Eq. 7 / r
    } else {
        f = (r > 0.f) ? c.vk * atanf(r * c.inv_rt) / r : c.vk * c.inv_rt;        // Eq. 6 / r
    }
    return c.vsys + f * xe * c.sin_i;
}

constexpr int kVfRanks = 8;                     // groups of 32 chains = CTAs of a cluster
constexpr int kVfSteps = kVfThreads / 32;       // steps of a chain evaluated at once = warps

// A pixel's maps and residuals; returns its share of chi2.
__device__ __forceinline__ float vf_pixel(const FusedArgs &a, const VfConst &c, const gbk_obs &ob, int model, int pix)
{
    const int nx = a.g.nx, np = a.g.nx * a.g.ny;
    const float nanf_ = __int_as_float(0x7fc00000);
    const int y = pix / nx, x = pix - y * nx;
    float m1 = c.valid ? vf_velocity(c, (float)x, (float)y) : nanf_;
    float m2 = c.valid ? c.sig0 : nanf_;
    float m0 = c.valid ? 1.f : nanf_;
    if (a.maps) {
        float *mp = a.maps + (size_t)model * 3 * np;
        mp[pix] = m0;
        mp[np + pix] = m1;
        mp[2 * np + pix] = m2;
    }
    if (!a.chi2 && !a.resid) return 0.f;
    float rv = 0.f, rs = 0.f;
    if (ob.mask[pix] != 0) {
        rv = ob.w_v[pix] * (m1 - ob.v_obs[pix]);
        rs = ob.w_s[pix] * (m2 - ob.s_obs[pix]);
    }
    if (a.resid) {
        float *rp = a.resid + (size_t)model * 2 * np;
        rp[pix] = rv;
        rp[np + pix] = rs;
    }
    return __fmaf_rn(rv, rv, __fmul_rn(rs, rs));  // spelt out: the same bits from both kernels
}

// The next term of a chain (Kahan).
__device__ __forceinline__ void vf_add(float t2, float &s, float &comp)
{
    float yk = t2 - comp, tk = s + yk;
    comp = (tk - s) - yk;
    s = tk;
}

__global__ void __cluster_dims__(kVfRanks, 1, 1) __launch_bounds__(kVfThreads) vfield_kernel(FusedArgs a)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    __shared__ VfConst s_c;
    __shared__ gbk_obs s_ob;
    __shared__ float term[2][kVfSteps][32];
    __shared__ double red[kVfRanks];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int np = a.g.nx * a.g.ny;
    const int mpg = a.models_per_gal;
    const int first = rank * 32 + lane;  // the chain's first pixel
    cluster.sync();  // every CTA has started: its shared memory may be written
    const int model = blockIdx.x / kVfRanks, gal = mpg > 0 ? model / mpg : 0;
    if (a.skip && a.skip[gal] != 0) return;  // the whole cluster
    if (tid == 0) {
        s_c = vf_const(a.params + (size_t)model * GBK_NPAR, a.g.model);
        s_ob = a.obs_list ? a.obs_list[gal] : a.obs;
    }
    __syncthreads();
    const VfConst c = s_c;
    float s = 0.f, comp = 0.f;  // warp 0
    int buf = 0;
    for (int base = 0; rank * 32 + base < np; base += kVfThreads * kVfSteps, buf ^= 1) {
        const int pix = first + base + warp * kVfThreads;
        if (pix < np) term[buf][warp][lane] = vf_pixel(a, c, s_ob, model, pix);
        if (!a.chi2) continue;
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int k = 0; k < kVfSteps; ++k) {
                if (first + base + k * kVfThreads >= np) break;
                vf_add(term[buf][k][lane], s, comp);
            }
        }
    }
    if (!a.chi2) return;
    // the chains' sum in FP32 (a fixed shuffle tree), the groups in FP64
    if (warp == 0) {
        float v = s - comp;
        for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
        if (lane == 0) *cluster.map_shared_rank(&red[rank], 0) = (double)v;
    }
    cluster.sync();
    if (rank == 0 && tid == 0) {
        double tot = 0.0;
        for (int w = 0; w < kVfRanks; ++w) tot += red[w];
        a.chi2[model] = c.valid ? tot : (double)__int_as_float(0x7fc00000);
    }
}

// The same with one CTA per model and a thread per chain.
__global__ void __launch_bounds__(kVfThreads) vfield_many_kernel(FusedArgs a)
{
    __shared__ VfConst s_c;
    __shared__ gbk_obs s_ob;
    __shared__ double red[kVfRanks];
    const int tid = threadIdx.x;
    const int np = a.g.nx * a.g.ny;
    const int mpg = a.models_per_gal;
    for (int model = blockIdx.x; model < a.n_models; model += gridDim.x) {
        const int gal = mpg > 0 ? model / mpg : 0;
        if (a.skip && a.skip[gal] != 0) continue;
        if (tid == 0) {
            s_c = vf_const(a.params + (size_t)model * GBK_NPAR, a.g.model);
            s_ob = a.obs_list ? a.obs_list[gal] : a.obs;
        }
        __syncthreads();
        const VfConst c = s_c;
        float s = 0.f, comp = 0.f;
        for (int pix = tid; pix < np; pix += kVfThreads) vf_add(vf_pixel(a, c, s_ob, model, pix), s, comp);
        if (a.chi2) {
            float v = s - comp;
            for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
            if ((tid & 31) == 0) red[tid >> 5] = (double)v;
            __syncthreads();
            if (tid == 0) {
                double tot = 0.0;
                for (int w = 0; w < kVfRanks; ++w) tot += red[w];
                a.chi2[model] = c.valid ? tot : (double)__int_as_float(0x7fc00000);
            }
        }
        __syncthreads();  // s_c, s_ob and red are rewritten by the next model
    }
}

// ---------------------------------------------------------------------------
// Analytic Jacobian of the velocity-field residuals.  With F(r) = Vrot(r) / r,
// m1 = Vsys + F(r) x_e sin i and m2 = sigma0; by the chain rule through
// Eqs. 1-4 (angles in degrees):
//   d x_e = (sin PA, -cos PA, y_e k)  and  d y_e = (cos PA, sin PA, -x_e k)
//   for (x0, y0, PA), k = pi / 180;  d y_d = d y_e / cos i, and for the
//   inclination d y_d / di = y_d tan i k;  d r = (x_e dx_e + y_d dy_d) / r;
//   dm1 = sin i (F'(r) dr x_e + F dx_e) for (x0, y0, PA),
//   dm1/di = F x_e cos i k + sin i F'(r) dr_i x_e,  dm1/dVsys = 1,
//   dm1/dtheta = sin i x_e dF/dtheta for the curve's parameters;
//   arctan (Eq. 6, c = 2 Vmax / pi, u = r / r_t):
//     F' = c (u / (1 + u^2) - atan u) / r^2 (series for small u),
//     dF/dVmax = (2 / pi) atan(u) / r,  dF/dr_t = -c / (r_t^2 + r^2);
//   Epinat (Eq. 7, q = r / r_t, D = 1 + q^a):
//     F' = (F / r) ((g - 1) - a q^a / D),  dF/dV_t = q^g / (D r),
//     dF/dr_t = -(F / r_t) (g - a q^a / D),  dF/da = -F q^a ln q / D,
//     dF/dg = F ln q;
//   dm2/dsigma0 = 1.  At r = 0 the cusp of r gets the one-sided value 0 (and
//   the Epinat curve, whose F is 0 there, zero derivatives).  Rows are
//   J_v = w_v dm1, J_s = w_s dm2 on unmasked pixels; J^T J, J^T v and sum r^2
//   of all ten parameters are summed over the chains in the order above.
constexpr int kVfEnt = GBK_NPAR * (GBK_NPAR + 1) / 2 + GBK_NPAR + 1;
// A pixel's terms: J_v for nine parameters (the dispersion has none), J_s of
// the dispersion, the cotangent and the residuals of the two maps.
constexpr int kVfRec = 14, kVfWs = 9, kVfCv = 10, kVfCs = 11, kVfRv = 12, kVfRs = 13;
__host__ __device__ constexpr int vf_slot(int k) { return k < GBK_SIG0 ? k : k - 1; }

// Warp WARP's share of the entries (J^T J upper triangle, J^T v, sum r^2) over
// the steps at hand, in the chains' order; rec = [step][kVfRec][32].
template <int WARP>
__device__ __forceinline__ void vf_accumulate(const float *rec, int steps, int lane, float (&E)[(kVfEnt + 7) / 8])
{
    constexpr int e0 = WARP * kVfEnt / 8, e1 = (WARP + 1) * kVfEnt / 8;
    for (int s = 0; s < steps; ++s) {
        const float *const q = rec + s * kVfRec * 32 + lane;
        int e = 0;
#pragma unroll
        for (int j = 0; j < GBK_NPAR; ++j)
#pragma unroll
            for (int k = j; k < GBK_NPAR; ++k, ++e) {
                if (e < e0 || e >= e1) continue;
                const float vj = j == GBK_SIG0 ? 0.f : q[32 * vf_slot(j)], vk = k == GBK_SIG0 ? 0.f : q[32 * vf_slot(k)];
                const float sj = j == GBK_SIG0 ? q[32 * kVfWs] : 0.f, sk = k == GBK_SIG0 ? q[32 * kVfWs] : 0.f;
                E[e - e0] = fmaf(vj, vk, fmaf(sj, sk, E[e - e0]));
            }
#pragma unroll
        for (int j = 0; j < GBK_NPAR; ++j, ++e) {
            if (e < e0 || e >= e1) continue;
            const float vj = j == GBK_SIG0 ? 0.f : q[32 * vf_slot(j)], sj = j == GBK_SIG0 ? q[32 * kVfWs] : 0.f;
            E[e - e0] = fmaf(vj, q[32 * kVfCv], fmaf(sj, q[32 * kVfCs], E[e - e0]));
        }
        if (e >= e0 && e < e1)
            E[e - e0] = fmaf(q[32 * kVfRv], q[32 * kVfRv], fmaf(q[32 * kVfRs], q[32 * kVfRs], E[e - e0]));
    }
}

// A pixel's Jacobian rows (jv of the velocity, js of the dispersion; written to
// `jac` too), cotangent and residuals.
__device__ __forceinline__ void vf_pixel_rows(const TangentArgs &a, const VfConst &c, const gbk_obs &ob, float vmax,
                                              int model, int pix, float (&jv)[GBK_NPAR], float (&js)[GBK_NPAR],
                                              float &cv, float &cs, float &rv, float &rs)
{
    const int nx = a.g.nx, np = a.g.nx * a.g.ny;
    const float kdeg = 0.017453292519943295f;
    const float si = c.sin_i, ci = 1.f / c.inv_cos_i, ti = si * c.inv_cos_i;
    const int y = pix / nx, x = pix - y * nx;
    float dx = (float)x - c.x0, dy = (float)y - c.y0;
    float xe = -dx * c.sin_pa + dy * c.cos_pa;
    float ye = -dx * c.cos_pa - dy * c.sin_pa;
    float yd = ye * c.inv_cos_i;
    float r = sqrtf(xe * xe + yd * yd);
    float F, Fr, Fv, Frt, Fa = 0.f, Fg = 0.f;
    if (c.epinat) {
        if (r > 0.f) {
            float q = r * c.inv_rt, lq = logf(q);
            float qg = expf(c.g * lq), qa = expf(c.a * lq), D = 1.f + qa;
            Fv = qg / (D * r);
            F = c.vk * Fv;
            float aq = c.a * qa / D;
            Fr = F / r * ((c.g - 1.f) - aq);
            Frt = -F * c.inv_rt * (c.g - aq);
            Fa = -F * qa * lq / D;
            Fg = F * lq;
        } else {
            F = Fr = Fv = Frt = 0.f;
        }
    } else {
        float u = r * c.inv_rt, at = atanf(u);
        Fv = 0.63661977f * ((r > 0.f) ? at / r : c.inv_rt);
        F = vmax * Fv;
        if (r <= 0.f) Fr = 0.f;
        else if (u < 0.1f) Fr = c.vk * c.inv_rt * c.inv_rt * u * (-2.f / 3.f + 0.8f * u * u);
        else Fr = c.vk * (u / (1.f + u * u) - at) / (r * r);
        float rt = 1.f / c.inv_rt;
        Frt = -c.vk / (rt * rt + r * r);
    }
    float m1 = c.vsys + F * xe * si;
    float rx = 0.f, ry = 0.f, ri = 0.f;  // dr per unit dx_e, dy_e; dr/di
    if (r > 0.f) {
        rx = xe / r;
        ry = yd * c.inv_cos_i / r;
        ri = yd * yd * ti * kdeg / r;
    }
#pragma unroll
    for (int k = 0; k < GBK_NPAR; ++k) { jv[k] = 0.f; js[k] = 0.f; }
    rv = rs = cv = cs = 0.f;
    if (c.valid && ob.mask[pix] != 0) {
        const float wv = ob.w_v[pix], ws = ob.w_s[pix];
        const float dxe[3] = {c.sin_pa, -c.cos_pa, ye * kdeg};
        const float dye[3] = {c.cos_pa, c.sin_pa, -xe * kdeg};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float dr = rx * dxe[k] + ry * dye[k];
            jv[k] = wv * si * (Fr * dr * xe + F * dxe[k]);
        }
        jv[GBK_INCL] = wv * (F * xe * ci * kdeg + si * Fr * ri * xe);
        jv[GBK_VSYS] = wv;
        jv[GBK_VMAX] = wv * si * xe * Fv;
        jv[GBK_RT] = wv * si * xe * Frt;
        jv[GBK_EPI_A] = wv * si * xe * Fa;
        jv[GBK_EPI_G] = wv * si * xe * Fg;
        js[GBK_SIG0] = ws;
        rv = wv * (m1 - ob.v_obs[pix]);
        rs = ws * (c.sig0 - ob.s_obs[pix]);
        if (a.cot) {
            cv = a.cot[(size_t)model * 2 * np + pix];
            cs = a.cot[(size_t)model * 2 * np + np + pix];
        } else {
            cv = rv;
            cs = rs;
        }
    }
    if (a.jac) {
        float *J = a.jac + (size_t)model * GBK_NPAR * 2 * np;
#pragma unroll
        for (int k = 0; k < GBK_NPAR; ++k) {
            J[((size_t)k * 2) * np + pix] = jv[k];
            J[((size_t)k * 2 + 1) * np + pix] = js[k];
        }
    }
}

// A model's outputs from its sums of all ten parameters (the whole block).
__device__ __forceinline__ void vf_write(const TangentArgs &a, const double *s_part, bool valid, int model, int tid)
{
    const int nf = a.np, ntri = nf * (nf + 1) / 2;
    if (tid < ntri + nf + 1) {
        int src, j = 0, k = 0;
        if (tid < ntri) {
            int t = tid;
            while (t >= nf - j) { t -= nf - j; ++j; }
            k = j + t;
            int p = a.free_idx[j], q = a.free_idx[k];
            if (p > q) { int w = p; p = q; q = w; }
            src = p * GBK_NPAR - p * (p - 1) / 2 + (q - p);
        } else if (tid < ntri + nf) {
            src = GBK_NPAR * (GBK_NPAR + 1) / 2 + a.free_idx[tid - ntri];
        } else {
            src = kVfEnt - 1;
        }
        double v = valid ? s_part[src] : (double)__int_as_float(0x7fc00000);
        if (tid < ntri) {
            if (a.jtj) {
                a.jtj[(size_t)model * nf * nf + j * nf + k] = v;
                a.jtj[(size_t)model * nf * nf + k * nf + j] = v;
            }
        } else if (tid < ntri + nf) {
            if (a.jtv) a.jtv[(size_t)model * nf + (tid - ntri)] = v;
        } else if (a.chi2) {
            a.chi2[model] = v;
        }
    }
}

__global__ void __cluster_dims__(kVfRanks, 1, 1) __launch_bounds__(kVfThreads) vfield_tangent_kernel(TangentArgs a)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    __shared__ VfConst s_c;
    __shared__ gbk_obs s_ob;
    __shared__ float rec[2][kVfSteps][kVfRec][32];
    __shared__ float wred[kVfRanks][kVfEnt];  // the groups' sums (rank 0's copy is used)
    __shared__ double s_part[kVfEnt];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int np = a.g.nx * a.g.ny;
    const int mpg = a.models_per_gal;
    const int first = rank * 32 + lane;  // the chain's first pixel
    cluster.sync();  // every CTA has started: its shared memory may be written
    const int model = blockIdx.x / kVfRanks, gal = mpg > 0 ? model / mpg : 0;
    if (a.skip && a.skip[gal] != 0) return;  // the whole cluster
    if (tid == 0) {
        s_c = vf_const(a.params + (size_t)model * GBK_NPAR, a.g.model);
        s_ob = a.obs_list ? a.obs_list[gal] : a.obs;
    }
    __syncthreads();
    const VfConst c = s_c;
    const float vmax = (float)a.params[(size_t)model * GBK_NPAR + GBK_VMAX];
    float E[(kVfEnt + 7) / 8];
#pragma unroll
    for (int e = 0; e < (kVfEnt + 7) / 8; ++e) E[e] = 0.f;
    int buf = 0;
    for (int base = 0; rank * 32 + base < np; base += kVfThreads * kVfSteps, buf ^= 1) {
        const int pix = first + base + warp * kVfThreads;
        if (pix < np) {
            float jv[GBK_NPAR], js[GBK_NPAR], cv, cs, rv, rs;
            vf_pixel_rows(a, c, s_ob, vmax, model, pix, jv, js, cv, cs, rv, rs);
            float *const o = &rec[buf][warp][0][lane];
#pragma unroll
            for (int k = 0; k < GBK_NPAR; ++k)
                if (k != GBK_SIG0) o[32 * vf_slot(k)] = jv[k];
            o[32 * kVfWs] = js[GBK_SIG0];
            o[32 * kVfCv] = cv;
            o[32 * kVfCs] = cs;
            o[32 * kVfRv] = rv;
            o[32 * kVfRs] = rs;
        }
        __syncthreads();
        // the chain's steps at hand that exist
        int steps = (np - 1 - first - base) / kVfThreads + 1;
        steps = first + base >= np ? 0 : min(steps, kVfSteps);
        const float *const r = &rec[buf][0][0][0];
        switch (warp) {
        case 0: vf_accumulate<0>(r, steps, lane, E); break;
        case 1: vf_accumulate<1>(r, steps, lane, E); break;
        case 2: vf_accumulate<2>(r, steps, lane, E); break;
        case 3: vf_accumulate<3>(r, steps, lane, E); break;
        case 4: vf_accumulate<4>(r, steps, lane, E); break;
        case 5: vf_accumulate<5>(r, steps, lane, E); break;
        case 6: vf_accumulate<6>(r, steps, lane, E); break;
        default: vf_accumulate<7>(r, steps, lane, E); break;
        }
    }
    // the chains' sums in FP32 (a butterfly), the groups in FP64 in order
    const int e0 = warp * kVfEnt / 8, e1 = (warp + 1) * kVfEnt / 8;
#pragma unroll
    for (int i = 0; i < (kVfEnt + 7) / 8; ++i) {
        float v = E[i];
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0 && e0 + i < e1) *cluster.map_shared_rank(&wred[rank][e0 + i], 0) = v;
    }
    cluster.sync();
    if (rank != 0) return;
    for (int e = tid; e < kVfEnt; e += kVfThreads) {
        double v = 0.0;
        for (int q = 0; q < kVfRanks; ++q) v += (double)wred[q][e];
        s_part[e] = v;
    }
    __syncthreads();
    vf_write(a, s_part, c.valid, model, tid);
}

// The same with one CTA per model and a thread per chain, all entries in its
// registers.
__global__ void __launch_bounds__(kVfThreads) vfield_tangent_many_kernel(TangentArgs a)
{
    __shared__ VfConst s_c;
    __shared__ gbk_obs s_ob;
    __shared__ float wred[kVfRanks][kVfEnt];
    __shared__ double s_part[kVfEnt];
    const int tid = threadIdx.x;
    const int np = a.g.nx * a.g.ny;
    const int mpg = a.models_per_gal;
    for (int model = blockIdx.x; model < a.n_models; model += gridDim.x) {
        const int gal = mpg > 0 ? model / mpg : 0;
        if (a.skip && a.skip[gal] != 0) continue;
        if (tid == 0) {
            s_c = vf_const(a.params + (size_t)model * GBK_NPAR, a.g.model);
            s_ob = a.obs_list ? a.obs_list[gal] : a.obs;
        }
        __syncthreads();
        const VfConst c = s_c;
        const float vmax = (float)a.params[(size_t)model * GBK_NPAR + GBK_VMAX];
        float E[kVfEnt];
#pragma unroll
        for (int e = 0; e < kVfEnt; ++e) E[e] = 0.f;
        for (int pix = tid; pix < np; pix += kVfThreads) {
            float jv[GBK_NPAR], js[GBK_NPAR], cv, cs, rv, rs;
            vf_pixel_rows(a, c, s_ob, vmax, model, pix, jv, js, cv, cs, rv, rs);
            int e = 0;
#pragma unroll
            for (int j = 0; j < GBK_NPAR; ++j)
#pragma unroll
                for (int k = j; k < GBK_NPAR; ++k, ++e) E[e] = fmaf(jv[j], jv[k], fmaf(js[j], js[k], E[e]));
#pragma unroll
            for (int j = 0; j < GBK_NPAR; ++j, ++e) E[e] = fmaf(jv[j], cv, fmaf(js[j], cs, E[e]));
            E[e] = fmaf(rv, rv, fmaf(rs, rs, E[e]));
        }
        // the chains' sums in FP32 (a reduce-scatter), the groups in FP64 in order
        warp_sum_scatter<kVfEnt>(E, tid & 31, wred[tid >> 5]);
        __syncthreads();
        for (int e = tid; e < kVfEnt; e += kVfThreads) {
            double v = 0.0;
            for (int q = 0; q < kVfRanks; ++q) v += (double)wred[q][e];
            s_part[e] = v;
        }
        __syncthreads();
        vf_write(a, s_part, c.valid, model, tid);
        __syncthreads();  // s_c, s_ob, wred and s_part are rewritten by the next model
    }
}

// The largest batch that takes a cluster per model.  `alone`: for a call whose
// models all run.  A fit's finished ones only return (a.skip), and its long
// tail has few running, so there the line lies higher: fits of 512 fields of
// 256 x 256 take 18.7 ms with clusters and 24.7 without, 300 of 128 x 128 12.6
// and 13.3, 2048 of 64 x 64 17.7 and 14.4, 4096 of 48 x 48 24.0 and 15.3.
static long vf_cluster_models(const Geom &g, const int32_t *skip, long alone)
{
    return skip ? std::max(alone, (long)g.nx * g.ny / 48) : alone;
}

gbk_status launch_vfield_tangent(const TangentArgs &a, cudaStream_t st)
{
    if (a.geoms) return fail(GBK_EUNSUPPORTED, "survey batches serve the intensity-cube model");
    if (a.np < 1 || a.np > GBK_NPAR) return fail(GBK_EINVAL, "velocity-field Jacobian: bad free-parameter count");
    if (a.n_models <= 0) return GBK_OK;
    // A cluster per model while its CTAs find SMs of their own and the image
    // pays for the exchange of records: 152 fields of 128 x 128 72 us against 74
    // with one CTA each, 200 of them 94 against 86; 64 of 64 x 64 23 and 23, 128
    // of them 33 against 23; 200 of 256 x 256 307 against 328, 304 of them 458
    // against 329.
    if (a.n_models > vf_cluster_models(a.g, a.skip, std::min((long)a.g.nx * a.g.ny / 64,
                                                             (long)a.g.nx * a.g.ny >= 32768 ? 208l : 152l)))
        vfield_tangent_many_kernel<<<std::min(a.n_models, 152 * 8), kVfThreads, 0, st>>>(a);
    else
        vfield_tangent_kernel<<<a.n_models * kVfRanks, kVfThreads, 0, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "velocity-field Jacobian launch");
    return GBK_OK;
}

gbk_status launch_vfield(const FusedArgs &a, cudaStream_t st)
{
    if (a.geoms) return fail(GBK_EUNSUPPORTED, "survey batches serve the intensity-cube model");
    if (a.n_models <= 0) return GBK_OK;
    // as above; only chi2's terms are exchanged here: 152 fields of 64 x 64 14
    // us against 16, 200 of them 20 against 16; 200 of 128 x 128 39 against 48,
    // 304 of them 53 against 49
    if (a.n_models > vf_cluster_models(a.g, a.skip, (long)a.g.nx * a.g.ny >= 8192 ? 300 : 152))
        vfield_many_kernel<<<std::min(a.n_models, 152 * 16), kVfThreads, 0, st>>>(a);
    else
        vfield_kernel<<<a.n_models * kVfRanks, kVfThreads, 0, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "velocity-field kernel launch");
    return GBK_OK;
}

}  // namespace gbk
