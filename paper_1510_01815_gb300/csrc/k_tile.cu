// k_tile.cu -- the folded forward model (cube -> PSF x LSF convolution ->
// moments -> masked chi-squared, Sec. 2.2.2-2.2.6 of Bekiaris et al. 2015) in
// one kernel: one CTA takes a model's image (or a tile of it) from its
// parameters to its maps, residuals and chi2, with nothing in global memory
// in between.
//
// Phases of a CTA, all in shared memory:
//   lines   every spaxel of the tile extended by the PSF radius: geometry and
//           the folded line sums (q0, q1, q2) about their centre a
//           (line_table.cuh: closed form or polynomials, no channel loop);
//   x pass  four outputs of two rows per thread from the 4 + 2R columns they
//           share, in place: a round's threads read, meet at a barrier, and
//           write over the row's first columns (a task writes columns that no
//           later task of the row reads, so one barrier per round suffices);
//   y pass  four rows of two columns per thread, the moments, residuals and
//           the CTA's part of chi2.
// The four planes (q0, q1, q2, a) are stored by row pairs,
// [row pair][plane][column][2 rows] before the x pass and
// [row pair][plane][column pair][row][2 columns] after it, so that every
// 16-byte access carries two inputs of a pass for two lanes of f32x2
// arithmetic.  The PSF passes accumulate about a reference velocity of each
// group of four outputs (fused_line.cuh, about_ref); groups start at
// multiples of four spaxels whatever the tiling, so the maps do not depend on
// it.
//
// The grid is one resident wave; a CTA loops over its items (models or
// tiles).  The geometry's tables are made once per CTA; warp 0 sets up the
// next model while the others are in the y pass.  Where an image is cut into
// tiles the last CTA of a model (an arrival counter, reset by it) adds their
// chi2 parts in tile order.
//
// What bounds it: issue slots (51 % busy) and shared-memory wavefronts (60 %).
// Two CTAs of 384 threads an SM leave 80 registers a thread, and no instance
// fits them: 136 - 276 bytes a thread go to local memory and 160 - 408 come
// back, most of them around the PSF passes.
#include <algorithm>

#include "gbk_api_internal.h"
#include "k_tile.h"
#include "line_table.cuh"

namespace gbk {

constexpr int kTileThreads = 384;  // largest CTA; two of them fill an SM's registers at 80 a thread
constexpr int kTileMaxSmem = 225 * 1024;
constexpr int kNO = 4;             // outputs of a PSF task along the pass

struct TileArgs {
    Geom g;
    const double *params;    // [n_models][GBK_NPAR]
    gbk_obs obs;
    const gbk_obs *obs_list; // per galaxy (model m0 + i is galaxy (m0 + i) / mpg), or null: obs for all
    const int32_t *skip;     // per galaxy: non-zero = leave the galaxy's models alone (or null)
    int m0, mpg;
    float *maps;             // [n_models][3][ny][nx] or null
    double *chi2;            // [n_models] or null
    float *resid;            // [n_models][2][ny][nx] or null
    double *part;            // [n_models][tiles]
    unsigned *arrived;       // [n_models]
    int tx, ty, tiles_x, tiles;
    int items;               // models x tiles
    int vec;                 // rows of maps and resid start on 8-byte boundaries
};

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_approx(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// i = q n + r for 0 <= i <= 1024 and n >= 1 (one reciprocal; i + 1/2 is never
// within rounding of a multiple of n).
__device__ __forceinline__ void split_index(int i, int n, int &q, int &r)
{
    q = (int)(((float)i + 0.5f) * rcp_approx((float)n));
    r = i - q * n;
}

// model_const by a warp: lane k has parameter v (1 beyond the last), so the
// checks, the two sincospi and the five reciprocals each take one step
// instead of ten in a row.  The values are model_const's.
__device__ inline void model_const_warp(double v, const Geom &g, int lane, ModelConst &c)
{
    bool okl = isfinite(v);
    if (lane == GBK_INCL) okl = okl && v >= 0.0 && v < 90.0;
    if (lane == GBK_RT || lane == GBK_SIG0 || lane == GBK_I0 || lane == GBK_H) okl = okl && v > 0.0;
    const bool okw = __all_sync(0xffffffffu, okl);
    const float f = (float)v;
    float sn, cs;
    sincospif((float)(v * (1.0 / 180.0)), &sn, &cs);  // used by the angles
    float den = f;
    if (lane == GBK_INCL) den = cs;
    if (lane == GBK_SIG0 && g.lsf_mode == 1) den = sqrtf(f * f + g.sig_lsf_kms * g.sig_lsf_kms);
    const float inv = 1.f / den;
    switch (lane) {
    case GBK_X0: c.x0 = f; break;
    case GBK_Y0: c.y0 = f; break;
    case GBK_PA: c.sin_pa = sn; c.cos_pa = cs; break;
    case GBK_INCL: c.sin_i = sn; c.inv_cos_i = inv; break;
    case GBK_VSYS: c.vsys = f; break;
    case GBK_VMAX: c.vrot_k = (float)(0.63661977236758134 * v); break;
    case GBK_RT: c.inv_rt = inv; break;
    case GBK_SIG0:
        c.sigma = den;
        c.amp = g.dv / (den * 2.5066282746310002f);
        c.alpha = 0.84932180028801904f / den;
        break;
    case GBK_I0: c.i0 = f; break;
    case GBK_H: c.inv_h = inv; break;
    case 31: c.valid = okw ? 1 : 0; break;
    }
    __syncwarp();
}

// A tile's place and sizes.
struct TileDims {
    int model, tile, tx0, ty0, nxo, nyo;
    int npx, npy;    // output pairs along x and y
    int nrp, exw;    // extended row pairs and columns
    int PP, RP;      // floats of a plane of a row pair, and of a row pair (padded: see the x pass)
};

__device__ __forceinline__ TileDims tile_dims(const Geom &g, int R, int tx, int ty, int tiles_x, int model, int tile)
{
    TileDims d;
    d.model = model;
    d.tile = tile;
    const int tyi = tile / tiles_x, txi = tile - tyi * tiles_x;
    d.tx0 = txi * tx;
    d.ty0 = tyi * ty;
    d.nxo = min(tx, g.nx - d.tx0);
    d.nyo = min(ty, g.ny - d.ty0);
    d.npx = (d.nxo + 1) >> 1;
    d.npy = (d.nyo + 1) >> 1;
    d.nrp = d.npy + R;
    d.exw = 2 * (d.npx + R);
    d.PP = 2 * d.exw;
    d.RP = 4 * d.PP + 4;
    return d;
}

// One item (a tile of a model) in shared memory.
struct TileItem {
    TileDims d;
    ModelConst mc;
    LineCtx lc;
    LineTab lt;
    gbk_obs ob;
};

// An item from its model's parameters (one per lane), by one warp.
template <int R>
__device__ __forceinline__ void setup_item(const Geom &g, const TileArgs &a, int it, double p, int lane, float var_z,
                                           TileItem &m)
{
    model_const_warp(p, g, lane, m.mc);
    if (lane == 0) {
        m.lc = line_ctx(g, m.mc, var_z);
        m.lt = line_table_plan(g, m.mc, m.lc);
    } else if (lane == 1) {
        const int model = it / a.tiles;
        m.d = tile_dims(g, R, a.tx, a.ty, a.tiles_x, model, it - model * a.tiles);
        m.ob = a.obs_list ? a.obs_list[(a.m0 + model) / a.mpg] : a.obs;
    }
}

// The first of the items it, it + step, .. whose galaxy is not skipped.
__device__ __forceinline__ int next_item(const TileArgs &a, int it, int step, int end)
{
    if (a.skip)
        while (it < end && a.skip[(a.m0 + it / a.tiles) / a.mpg] != 0) it += step;
    return it;
}

// about_ref and shift_sums (fused_line.cuh) on two lanes; nref = minus the
// reference velocity.
__device__ __forceinline__ f32x2 neg2(f32x2 v)
{
    float lo, hi;
    upk2(v, lo, hi);
    return pk2(-lo, -hi);
}
__device__ __forceinline__ void about_ref2(f32x2 q0, f32x2 q1, f32x2 q2, f32x2 a, f32x2 nref, f32x2 &l1, f32x2 &l2)
{
    const f32x2 d = add2(a, nref);
    l1 = fma2(d, q0, q1);
    l2 = fma2(d, add2(l1, q1), q2);  // d q0 + 2 q1 = l1 + q1
}
__device__ __forceinline__ void shift_sums2(f32x2 delta, f32x2 s0, f32x2 &s1, f32x2 &s2)
{
    const f32x2 nd = neg2(delta);
    const f32x2 t = fma2(nd, s0, s1);   // s1 - delta s0
    s2 = fma2(nd, add2(t, s1), s2);     // s2 - 2 delta s1 + delta^2 s0
    s1 = t;
}

// A tap, read where it is used: held in registers all taps would spill too.
__device__ __forceinline__ f32x2 lds_tap(uint32_t addr)
{
    f32x2 w;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(w) : "r"(addr));
    return w;
}

// Two columns' row pairs to two rows' column pairs, one 16-byte store.
__device__ __forceinline__ void store_turned(float *p, f32x2 x0, f32x2 x1)
{
    float a0, a1, b0, b1;
    upk2(x0, a0, a1);
    upk2(x1, b0, b1);
    *reinterpret_cast<float4 *>(p) = make_float4(a0, b0, a1, b1);
}

// Two neighbouring map values (`vec`: rows start on 8-byte boundaries).
__device__ __forceinline__ void store_pair(float *p, const float (&v)[2], bool two, int vec)
{
    if (two && vec) {
        *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
    } else {
        p[0] = v[0];
        if (two) p[1] = v[1];
    }
}

// A PSF task: from pairs of inputs along the pass (two per 16-byte load, the
// other axis in the lanes) the sums of kNO consecutive outputs about the
// first one's centre.  `load` gives the k-th pair of inputs of a plane.
template <int R, class Load>
__device__ __forceinline__ void psf_pass(const Load &load, uint32_t taps, f32x2 nref, f32x2 (&s)[kNO][3])
{
    constexpr int W = 2 * R + 1;
    f32x2 w[kNO];  // taps e, e - 1, .. of the current input
#pragma unroll
    for (int k = 0; k < R + kNO / 2; ++k) {
        const ulonglong2 v0 = load(k, 0), v1 = load(k, 1), v2 = load(k, 2), va = load(k, 3);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = 2 * k + h;
            const f32x2 q0 = h ? v0.y : v0.x;
            f32x2 l1, l2;
            about_ref2(q0, h ? v1.y : v1.x, h ? v2.y : v2.x, h ? va.y : va.x, nref, l1, l2);
#pragma unroll
            for (int o = kNO - 1; o > 0; --o) w[o] = w[o - 1];
            if (e < W) w[0] = lds_tap(taps + 8 * e);
#pragma unroll
            for (int o = 0; o < kNO; ++o) {
                const int j = e - o;
                if (j == 0) {
                    s[o][0] = mul2(w[o], q0);
                    s[o][1] = mul2(w[o], l1);
                    s[o][2] = mul2(w[o], l2);
                } else if (j > 0 && j < W) {
                    s[o][0] = fma2(w[o], q0, s[o][0]);
                    s[o][1] = fma2(w[o], l1, s[o][1]);
                    s[o][2] = fma2(w[o], l2, s[o][2]);
                }
            }
        }
    }
}

// The direct sums of the spaxels that lines_phase left (marked with NaN; every
// one where no form serves the model).  Each lane has its own channel window;
// shared by the lanes that happen to be there, it made the last bits depend on
// the tiling.  Out of line: beside the other phases its code costs models that
// never take it 1 % (2048 models of 32 x 32 x 64: 51.1 us, 50.7 us so).
static __device__ __noinline__ void lines_direct(const Geom &g, const TileItem &M, int R, const float *edge, float *pl)
{
    const int tid = threadIdx.x, nthr = blockDim.x;
    const bool all = line_table_empty(M.lt);
    const int exw = M.d.exw, PP = M.d.PP, RP = M.d.RP, ntl = M.d.nrp * exw, etl = edge_table_len(g);
    const float xb = (float)(M.d.tx0 - R), yb = (float)(M.d.ty0 - R), inv_i0 = 1.f / M.mc.i0;
    int x, rp, dx, drp;
    split_index(tid, exw, rp, x);
    split_index(nthr, exw, drp, dx);
#pragma unroll 1
    for (int idx = tid; idx < ntl; idx += nthr) {
        float *const o = pl + rp * RP + 2 * x;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            if (!all && !isnan(o[h])) continue;
            const float4 q = line_sums<false>(g, M.mc, M.lc, edge, edge + etl, edge + 2 * etl, xb + (float)x,
                                              yb + (float)(2 * rp + h));
            o[h] = q.x * inv_i0;
            o[PP + h] = q.y * inv_i0;
            o[2 * PP + h] = q.z * inv_i0;
            o[3 * PP + h] = q.w;
        }
        x += dx;
        rp += drp;
        if (x >= exw) {
            x -= exw;
            ++rp;
        }
    }
}

// The lines of the extended tile; task: column x of a row pair, two spaxels.
// Threads come back to the spaxels that neither form serves in a loop of their
// own: as a call from this loop the direct sum cost every model registers, and
// where all lines take it (narrow ones) a third of the call.
__device__ __forceinline__ void lines_phase(const Geom &g, const TileItem &M, int R, const float *edge,
                                            const float *ltab, float *pl, int tid, int nthr)
{
    bool left = true;
    if (!line_table_empty(M.lt)) {
        const int exw = M.d.exw, PP = M.d.PP, RP = M.d.RP, ntl = M.d.nrp * exw;
        const DiscConst dc = disc_const(M.mc);
        int x, rp, dx, drp;
        split_index(tid, exw, rp, x);
        split_index(nthr, exw, drp, dx);
        const float xb = (float)(M.d.tx0 - R), yb = (float)(M.d.ty0 - R);
        left = false;
        for (int idx = tid; idx < ntl; idx += nthr) {
            float4 q[2];
            line_sums_pair(dc, M.lc, M.lt, ltab, xb + (float)x, yb + (float)(2 * rp), q, left);
            float *o = pl + rp * RP + 2 * x;
            *reinterpret_cast<float2 *>(o) = make_float2(q[0].x, q[1].x);
            *reinterpret_cast<float2 *>(o + PP) = make_float2(q[0].y, q[1].y);
            *reinterpret_cast<float2 *>(o + 2 * PP) = make_float2(q[0].z, q[1].z);
            *reinterpret_cast<float2 *>(o + 3 * PP) = make_float2(q[0].w, q[1].w);
            x += dx;
            rp += drp;
            if (x >= exw) {
                x -= exw;
                ++rp;
            }
        }
    }
    if (left) lines_direct(g, M, R, edge, pl);
}

// The x pass; task: outputs 4 xq .. 4 xq + 3 of a row pair, rows in the lanes.
// Neighbouring threads take the two row pairs of a group in turn: with a row
// pair one 16-byte unit longer than a multiple of 32 bytes their loads (32
// bytes apart along x) fall on all banks.
template <int R>
__device__ __forceinline__ void x_phase(const TileItem &M, uint32_t taps, float *pl, int tid, int nthr)
{
    const int npx = M.d.npx, nrp = M.d.nrp, PP = M.d.PP, RP = M.d.RP;
    const int nq = (npx + 1) >> 1, ngr = (nrp + 1) >> 1;  // tasks of a row pair, groups of two row pairs
    int gr, r2, dgr, dr2;
    split_index(tid, 2 * nq, gr, r2);
    split_index(nthr, 2 * nq, dgr, dr2);
    for (int t0 = 0; t0 < ngr * 2 * nq; t0 += nthr) {
        const int rp = 2 * gr + (r2 & 1), xq = r2 >> 1;
        const bool on = rp < nrp;
        float *const b = pl + rp * RP + 8 * xq;
        f32x2 s[kNO][3], cen[kNO];
        if (on) {
            const f32x2 nref = neg2(*reinterpret_cast<const f32x2 *>(b + 3 * PP + 2 * R));
            psf_pass<R>([&](int k, int m) { return *reinterpret_cast<const ulonglong2 *>(b + m * PP + 4 * k); }, taps,
                        nref, s);
#pragma unroll
            for (int o = 0; o < kNO; ++o) {
                cen[o] = *reinterpret_cast<const f32x2 *>(b + 3 * PP + 2 * (R + o));
                if (o) shift_sums2(add2(cen[o], nref), s[o][0], s[o][1], s[o][2]);
            }
        }
        __syncthreads();
        if (on) {
            // columns in the lanes from here on
#pragma unroll
            for (int h = 0; h < kNO / 2; ++h) {
                if (h && 2 * xq + 1 >= npx) break;  // past the row's outputs
#pragma unroll
                for (int m = 0; m < 3; ++m) store_turned(b + m * PP + 4 * h, s[2 * h][m], s[2 * h + 1][m]);
                store_turned(b + 3 * PP + 4 * h, cen[2 * h], cen[2 * h + 1]);
            }
        }
        r2 += dr2;
        gr += dgr;
        if (r2 >= 2 * nq) {
            r2 -= 2 * nq;
            ++gr;
        }
    }
}

// The y pass; task: rows 4 yq .. 4 yq + 3 of a column pair, columns in the
// lanes; then the moments and residuals.  Returns the thread's sum of squared
// residuals.
template <int R>
__device__ __forceinline__ float y_phase(const TileItem &M, uint32_t taps, const float *pl, int nx, size_t np,
                                         float *maps, float *resid, bool want_obs, int vec, int tid, int nthr)
{
    const ModelConst &c = M.mc;
    const int npx = M.d.npx, nxo = M.d.nxo, nyo = M.d.nyo, PP = M.d.PP, RP = M.d.RP;
    const size_t pix0 = (size_t)M.d.ty0 * nx + M.d.tx0;
    const float nanf_ = __int_as_float(0x7fc00000);
    if (maps) maps += 3 * (size_t)M.d.model * np + pix0;
    if (resid) resid += 2 * (size_t)M.d.model * np + pix0;
    const float i0 = c.i0;  // the sums are per unit I0, so the approximations below see normal numbers
    KahanF acc;
    const int nyq = (M.d.npy + 1) >> 1;
    int yq, xp, dyq, dxp;
    split_index(tid, npx, yq, xp);
    split_index(nthr, npx, dyq, dxp);
    for (int t = tid; t < nyq * npx; t += nthr) {
        const float *const b = pl + 2 * yq * RP + 4 * xp;
        f32x2 s[kNO][3];
        const f32x2 nref = neg2(*reinterpret_cast<const f32x2 *>(b + (R >> 1) * RP + 3 * PP + 2 * (R & 1)));
        psf_pass<R>([&](int k, int m) { return *reinterpret_cast<const ulonglong2 *>(b + k * RP + m * PP); }, taps,
                    nref, s);
#pragma unroll
        for (int o = 0; o < kNO; ++o) {
            const int yl = 4 * yq + o, x = 2 * xp;
            if (yl >= nyo) break;
            const f32x2 cen = *reinterpret_cast<const f32x2 *>(b + ((R + o) >> 1) * RP + 3 * PP + 2 * ((R + o) & 1));
            if (o) shift_sums2(add2(cen, nref), s[o][0], s[o][1], s[o][2]);
            const bool two = x + 1 < nxo;
            const size_t po = (size_t)yl * nx + x;
            float m0[2], m1[2], m2[2], s0[2], s1[2], s2[2], ce[2];
            bool valid[2];
            upk2(s[o][0], s0[0], s0[1]);
            upk2(s[o][1], s1[0], s1[1]);
            upk2(s[o][2], s2[0], s2[1]);
            upk2(cen, ce[0], ce[1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                // __frcp_rn and sqrtf here cost 7 - 9 % of the whole call
                // (8192 images of 64 x 64: 482 -> 527 us) and move the
                // dispersion's error against 64 bits from 0.94 to 0.92 of what
                // it was with sampled lines, so the approximations stay
                valid[h] = s0[h] > kInvalidFraction;
                const float inv = rcp_approx(s0[h]), mu = s1[h] * inv;
                const float var = fmaf(-mu, mu, s2[h] * inv);
                m0[h] = valid[h] ? s0[h] * i0 : 0.f;
                m1[h] = valid[h] ? ce[h] + mu : c.vsys;
                m2[h] = valid[h] ? sqrt_approx(fmaxf(var, 0.f)) : 0.f;
                if (!c.valid) m0[h] = m1[h] = m2[h] = nanf_;
            }
            if (maps) {
                store_pair(maps + po, m0, two, vec);
                store_pair(maps + np + po, m1, two, vec);
                store_pair(maps + 2 * np + po, m2, two, vec);
            }
            if (want_obs) {
                const size_t pix = pix0 + po;
                float rv[2] = {0.f, 0.f}, rs[2] = {0.f, 0.f};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if ((h == 0 || two) && __ldg(M.ob.mask + pix + h) != 0 && (valid[h] || !c.valid)) {
                        rv[h] = __ldg(M.ob.w_v + pix + h) * (m1[h] - __ldg(M.ob.v_obs + pix + h));
                        rs[h] = __ldg(M.ob.w_s + pix + h) * (m2[h] - __ldg(M.ob.s_obs + pix + h));
                    }
                    acc.add_square(rv[h]);
                    acc.add_square(rs[h]);
                }
                if (resid) {
                    store_pair(resid + po, rv, two, vec);
                    store_pair(resid + np + po, rs, two, vec);
                }
            }
        }
        xp += dxp;
        yq += dyq;
        if (xp >= npx) {
            xp -= npx;
            ++yq;
        }
    }
    return acc.s - acc.c;
}

// The block's sum of squared residuals (thread 0): each warp's sum in FP32
// (the compensated per-thread sums, a fixed shuffle tree), the warps in FP64.
__device__ __forceinline__ double block_chi2(float v, double *red, int tid, int nthr)
{
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if ((tid & 31) == 0) red[tid >> 5] = (double)v;
    __syncthreads();
    double sum = 0.0;
    if (tid == 0)
        for (int k = 0; k < (nthr >> 5); ++k) sum += red[k];
    return sum;
}

// A tile's part of its model's chi2 (one thread of the block): the last of a
// model's tiles adds up all parts in tile order.
__device__ __forceinline__ void chi2_part(double sum, bool valid, int model, int tile, int tiles, double *chi2,
                                          double *part, unsigned *arrived)
{
    const double bad = (double)__int_as_float(0x7fc00000);
    if (tiles == 1) {
        chi2[model] = valid ? sum : bad;
        return;
    }
    part[(size_t)model * tiles + tile] = sum;
    __threadfence();
    if (atomicAdd(&arrived[model], 1u) == (unsigned)tiles - 1) {
        __threadfence();
        const volatile double *p = part + (size_t)model * tiles;
        double tot = 0.0;
        for (int k = 0; k < tiles; ++k) tot += p[k];
        chi2[model] = valid ? tot : bad;
        arrived[model] = 0u;  // ready for the next call
    }
}

// A geometry's taps, in shared memory.
struct TileTaps {
    f32x2 w2[2 * kTileMaxR + 1];  // normalised PSF taps, twice each
    float w[2 * kTileMaxR + 1], lz[2 * kMaxRadius + 1];
    float var;                    // LSF variance
};

// A geometry's taps, LSF variance and band-edge tables (fused_line.cuh,
// edge_tables) with the whole block (over a warp); ends with a barrier.
__device__ __forceinline__ void tile_tables(const Geom &g, int R, TileTaps &T, float *edge, int tid, int nthr)
{
    const int W = 2 * R + 1;
    const int lane = tid & 31, etl = edge_table_len(g);
    for (int j = tid; j <= 2 * g.Rz; j += nthr) T.lz[j] = tap_raw(j - g.Rz, g.sig_z, g.Rz);
    if (tid < W) T.w[tid] = tap_raw(tid - R, g.sig_xy, R);
    __syncthreads();
    if (tid < 32) {
        float S = 0.f, V = 0.f;
        for (int j = lane; j <= 2 * g.Rz; j += 32) {
            const float w = T.lz[j], d = (float)(j - g.Rz);
            S += w;
            V = fmaf(w * d, d, V);
        }
        for (int off = 16; off > 0; off >>= 1) {
            S += __shfl_xor_sync(0xffffffffu, S, off);
            V += __shfl_xor_sync(0xffffffffu, V, off);
        }
        if (lane == 0) T.var = g.dv * g.dv * (V / S);
        if (lane < W) {
            S = 0.f;
#pragma unroll
            for (int j = 0; j < 2 * kTileMaxR + 1; ++j)
                if (j < W) S += T.w[j];
            const float w = T.w[lane] / S;
            T.w2[lane] = pk2(w, w);
        }
    } else {
        const int elo = edge_lo_end(g), ehi = edge_hi_begin(g), hi_off = (elo + 1) & ~1;
        for (int k = tid - 32; k < elo + (g.ez - ehi); k += nthr - 32) {
            const bool lower = k < elo;
            const int e = lower ? k : ehi + (k - elo);
            const int kd = e - g.Rz;
            const int jlo = max(0, kd - g.Rz) - kd, jhi = min(g.nz - 1, kd + g.Rz) - kd;
            float Sz = 0.f, G0 = 0.f, H1 = 0.f, H2 = 0.f;
            for (int j = -g.Rz; j <= g.Rz; ++j) {
                const float w = T.lz[j + g.Rz];
                Sz += w;
                if (j >= jlo && j <= jhi) {
                    G0 += w;
                    H1 = fmaf(w, (float)j, H1);
                    H2 = fmaf(w, (float)(j * j), H2);
                }
            }
            G0 /= Sz;
            H1 = g.dv * (H1 / Sz);
            H2 = g.dv * g.dv * (H2 / Sz);
            const float eref = lower ? 0.5f * (float)(elo - 1) : 0.5f * (float)(ehi + g.ez - 1);
            const float delta = ((float)e - eref) * g.dv;
            const int slot = lower ? e : hi_off + (e - ehi);
            edge[slot] = G0;
            edge[etl + slot] = fmaf(delta, G0, H1);
            edge[2 * etl + slot] = fmaf(delta, fmaf(delta, G0, 2.f * H1), H2);
        }
    }
    __syncthreads();
}

// MULTI: models of several tiles (without it the loop keeps fewer values alive).
template <int R, bool MULTI>
__global__ void __launch_bounds__(kTileThreads, 2) tile_kernel(const __grid_constant__ TileArgs a)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ TileItem s_m[2];
    __shared__ TileTaps T;
    __shared__ double red[kTileThreads / 32];
    const Geom &g = a.g;
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
    const uint32_t taps = (uint32_t)__cvta_generic_to_shared(T.w2);
    const int etl = edge_table_len(g);
    float *const edge = sm, *const ltab = sm + 3 * etl, *const pl = ltab + kLtMaxSeg * kLtSegF;

    // One tile per model: the items in turn over the CTAs.  Several: a run of
    // neighbouring items each, so that a model is set up once for most of its
    // tiles (unless galaxies are skipped, whose runs would be uneven).
    const int tiles = MULTI ? a.tiles : 1;
    const bool runs = MULTI && !a.skip;
    const int step = runs ? 1 : (int)gridDim.x;
    const int end = runs ? (int)((long long)(blockIdx.x + 1) * a.items / gridDim.x) : a.items;
    int it = next_item(a, runs ? (int)((long long)blockIdx.x * a.items / gridDim.x) : (int)blockIdx.x, step, end);
    if (it >= end) return;  // the whole CTA

    // the geometry's tables: taps, LSF variance, band edges (fused_line.cuh, edge_tables)
    double pv = 1.0;
    if (tid < GBK_NPAR) pv = a.params[(size_t)(it / tiles) * GBK_NPAR + tid];
    tile_tables(g, R, T, edge, tid, nthr);
    if (tid < 32) setup_item<R>(g, a, it, pv, lane, T.var, s_m[0]);
    __syncthreads();

    const size_t np = (size_t)g.nx * g.ny;
    const bool want_chi2 = (a.chi2 != nullptr), want_obs = want_chi2 || a.resid;
    bool fresh = true;  // the slot's polynomials are still to be built
    for (int buf = 0; it < end;) {
        const TileItem &M = s_m[buf];
        const int nxt = next_item(a, it + step, step, end);
        const bool same = MULTI && nxt / tiles == it / tiles;  // a tile of the same model
        // the next model's parameters are on their way while this one runs
        if (tid < GBK_NPAR && nxt < end && !same) pv = a.params[(size_t)(nxt / tiles) * GBK_NPAR + tid];
        if (fresh && M.lt.nseg > 0) line_table_build(g, M.lc, M.lt, edge, etl, ltab, tid, nthr);
        lines_phase(g, M, R, edge, ltab, pl, tid, nthr);
        __syncthreads();
        x_phase<R>(M, taps, pl, tid, nthr);
        __syncthreads();
        // warp 0 sets up the next model before it joins the last pass
        if (tid < 32 && nxt < end && !same) setup_item<R>(g, a, nxt, pv, lane, T.var, s_m[buf ^ 1]);
        const float v = y_phase<R>(M, taps, pl, g.nx, np, a.maps, a.resid, want_obs, a.vec, tid, nthr);
        if (want_chi2) {
            const double sum = block_chi2(v, red, tid, nthr);
            if (tid == 0) chi2_part(sum, M.mc.valid, M.d.model, M.d.tile, tiles, a.chi2, a.part, a.arrived);
        }
        __syncthreads();  // the planes and the item slots change hands
        it = nxt;
        fresh = !same;
        if (same) {
            if (tid == 0) s_m[buf].d = tile_dims(g, R, a.tx, a.ty, a.tiles_x, it / tiles, it % tiles);
            __syncthreads();
        } else {
            buf ^= 1;
        }
    }
}

// chi2 from residuals, in the order in which tile_kernel adds them up in a
// given shape (a CTA per tile, its threads).  Calls with chi2 are bound to the
// shape of a large batch (TileShape); a small batch of large images leaves
// most SMs idle in it, so it takes the residuals in a shape of its own and then
// their sum here.  1 to 16 models of 128 x 128 x 64: 35 - 41 us in the large
// batch's shape, 24 - 29 us so.
struct ResidSumArgs {
    Geom g;
    const double *params;
    const float *resid;      // [n][2][ny][nx]
    const int32_t *skip;     // as TileArgs
    int m0, mpg;
    double *chi2, *part;
    unsigned *arrived;
    int tx, ty, tiles_x, tiles;
};

__global__ void __launch_bounds__(kTileThreads) tile_resid_sum_kernel(const ResidSumArgs a)
{
    __shared__ double red[kTileThreads / 32];
    const int model = blockIdx.x / a.tiles, tile = blockIdx.x - model * a.tiles;
    if (a.skip && a.skip[(a.m0 + model) / a.mpg] != 0) return;
    const int tid = threadIdx.x, nthr = blockDim.x, nx = a.g.nx;
    const size_t np = (size_t)nx * a.g.ny;
    const TileDims d = tile_dims(a.g, 0, a.tx, a.ty, a.tiles_x, model, tile);
    const float *r = a.resid + 2 * (size_t)model * np + (size_t)d.ty0 * nx + d.tx0;
    KahanF acc;
    const int nyq = (d.npy + 1) >> 1;
    for (int t = tid; t < nyq * d.npx; t += nthr) {  // y_phase's tasks and their order
        const int yq = t / d.npx, x = 2 * (t - yq * d.npx);
        float v[2 * kNO][2];
#pragma unroll
        for (int o = 0; o < kNO; ++o)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool in = 4 * yq + o < d.nyo && x + h < d.nxo;
                const float *q = r + (size_t)(4 * yq + o) * nx + x + h;
                v[2 * o + h][0] = in ? q[0] : 0.f;
                v[2 * o + h][1] = in ? q[np] : 0.f;
            }
#pragma unroll
        for (int o = 0; o < kNO; ++o) {
            if (4 * yq + o >= d.nyo) break;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                acc.add_square(v[2 * o + h][0]);
                acc.add_square(v[2 * o + h][1]);
            }
        }
    }
    const double sum = block_chi2(acc.s - acc.c, red, tid, nthr);
    if (tid != 0) return;
    const bool valid = model_const(a.params + (size_t)model * GBK_NPAR, a.g).valid;
    chi2_part(sum, valid, model, tile, a.tiles, a.chi2, a.part, a.arrived);
}

// Ragged batches: one galaxy's geometry per item, every image whole in one
// CTA, the items (costliest first) drawn from a work counter as the CTAs
// become free.  A launch has the CTA size that its largest galaxy's planes
// leave room for, 768 threads alone on an SM down to 160 with five on it, and
// galaxies of any PSF radius: launches by radius too were up to 45 in a row.
// The launches of a call overlap (programmatic dependent launch: the next one
// may start once this one's CTAs have, and none ends before the one before
// it has), so that one's last galaxies leave their SMs to the next one's first.
constexpr int kRaggedThreads = 768;

// Both PSF passes, the moments and residuals; the thread's sum of squares.
template <int R>
__device__ __forceinline__ float psf_phases(const TileItem &M, uint32_t taps, float *pl, int nx, size_t np,
                                            float *maps, float *resid, bool want_obs, int vec, int tid, int nthr)
{
    x_phase<R>(M, taps, pl, tid, nthr);
    __syncthreads();
    return y_phase<R>(M, taps, pl, nx, np, maps, resid, want_obs, vec, tid, nthr);
}

__global__ void __launch_bounds__(kRaggedThreads, 1) tile_ragged_kernel(const __grid_constant__ TileRagged a)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ TileItem M;
    __shared__ TileTaps T;
    __shared__ Geom g;
    __shared__ int s_item;
    __shared__ double red[kRaggedThreads / 32];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
    const uint32_t taps = (uint32_t)__cvta_generic_to_shared(T.w2);
    const bool want_chi2 = (a.chi2 != nullptr), want_obs = want_chi2 || a.resid;
    for (;;) {
        if (tid == 0) {
            int it;
            do {
                it = atomicAdd(a.work, 1);
            } while (it < a.items && a.skip && a.skip[a.order[it / a.mpg]] != 0);
            s_item = it;
            if (it < a.items) g = a.geoms[a.order[it / a.mpg]];
        }
        __syncthreads();
        const int it = s_item;
        if (it >= a.items) break;
        const int gal = a.order[it / a.mpg], sub = it % a.mpg;
        const size_t model = (size_t)gal * a.mpg + sub;
        const size_t np = (size_t)g.nx * g.ny, pix = (size_t)a.pix_off[gal] * a.mpg + (size_t)sub * np;
        const int etl = edge_table_len(g);
        float *const edge = sm, *const ltab = sm + 3 * etl, *const pl = ltab + kLtMaxSeg * kLtSegF;
        double pv = 1.0;
        if (tid < GBK_NPAR) pv = a.params[model * GBK_NPAR + tid];
        tile_tables(g, g.R, T, edge, tid, nthr);
        if (tid < 32) {
            model_const_warp(pv, g, lane, M.mc);
            if (lane == 0) {
                M.lc = line_ctx(g, M.mc, T.var);
                M.lt = line_table_plan(g, M.mc, M.lc);
            } else if (lane == 1) {
                M.d = tile_dims(g, g.R, g.nx, g.ny, 1, 0, 0);
                if (want_obs) M.ob = a.obs_list[gal];
            }
        }
        __syncthreads();
        if (M.lt.nseg > 0) line_table_build(g, M.lc, M.lt, edge, etl, ltab, tid, nthr);
        lines_phase(g, M, g.R, edge, ltab, pl, tid, nthr);
        __syncthreads();
        float *const maps = a.maps ? a.maps + 3 * pix : nullptr, *const resid = a.resid ? a.resid + 2 * pix : nullptr;
        const int vec = g.nx % 2 == 0 && ((uintptr_t)maps % 8) == 0 && ((uintptr_t)resid % 8) == 0;
        float v;
        switch (g.R) {  // the block's own
        case 0: v = psf_phases<0>(M, taps, pl, g.nx, np, maps, resid, want_obs, vec, tid, nthr); break;
        case 1: v = psf_phases<1>(M, taps, pl, g.nx, np, maps, resid, want_obs, vec, tid, nthr); break;
        case 2: v = psf_phases<2>(M, taps, pl, g.nx, np, maps, resid, want_obs, vec, tid, nthr); break;
        case 3: v = psf_phases<3>(M, taps, pl, g.nx, np, maps, resid, want_obs, vec, tid, nthr); break;
        case 4: v = psf_phases<4>(M, taps, pl, g.nx, np, maps, resid, want_obs, vec, tid, nthr); break;
        case 5: v = psf_phases<5>(M, taps, pl, g.nx, np, maps, resid, want_obs, vec, tid, nthr); break;
        case 6: v = psf_phases<6>(M, taps, pl, g.nx, np, maps, resid, want_obs, vec, tid, nthr); break;
        case 7: v = psf_phases<7>(M, taps, pl, g.nx, np, maps, resid, want_obs, vec, tid, nthr); break;
        default: v = psf_phases<8>(M, taps, pl, g.nx, np, maps, resid, want_obs, vec, tid, nthr); break;
        }
        if (want_chi2) {
            const double sum = block_chi2(v, red, tid, nthr);
            if (tid == 0) a.chi2[model] = M.mc.valid ? sum : (double)__int_as_float(0x7fc00000);
        }
        __syncthreads();
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");  // not before the launch before this one
}

// ---------------------------------------------------------------------------
// Host side.
static size_t tile_smem(const Geom &g, int tx, int ty)
{
    // output pairs along x; along y an even number (the last y task reads whole)
    const size_t npx = (std::min(tx, g.nx) + 1) / 2, npy = ((std::min(ty, g.ny) + 3) / 4) * 2;
    const size_t rp = 16 * (npx + g.R) + 4;  // floats of a row pair
    return ((npy + g.R) * rp + 3 * (size_t)edge_table_len(g) + (size_t)kLtMaxSeg * kLtSegF) * sizeof(float);
}

// CTAs of a shape that fit an SM: 3 KB of static and reserved shared memory
// each, 80 registers a thread.
static int tile_per_sm(size_t smem, int threads)
{
    return (int)std::min<size_t>(227 * 1024 / (smem + 3072), 800 / threads);
}

// Whole rounds of the CTA's threads: about 280 instructions a line task (two
// spaxels), 440 an x task and 740 a y task (eight outputs), 1500 of barriers
// and set-up.  An SM issues faster the more warps it holds, levelling off near
// 24.
double tile_cost(const Geom &g, const TileShape &s, int n_models)
{
    const double exw = s.tx + 2 * g.R, eyh = s.ty + 2 * g.R, nt = s.threads;
    const int per_sm = tile_per_sm(s.smem, s.threads);
    const double r1 = ceil(exw * eyh / 2 / nt), r2 = ceil(eyh / 2 * (s.tx / 4) / nt),
                 r3 = ceil((double)s.tx / 2 * (s.ty / 4) / nt);
    const double cta = 1500.0 + 280.0 * r1 + 440.0 * r2 + 740.0 * r3;
    const double ctas = (double)s.tiles * n_models;
    const double rounds = ceil(ctas / (152.0 * per_sm));
    const double warps = std::min(ceil(ctas / 152.0), (double)per_sm) * nt / 32;
    return rounds * cta * (10.0 + warps);
}

// The shapes of recent calls of this thread (the search takes longer than a
// small call's kernel).
struct ShapeKey {
    int nx, ny, R, etl, n, whole;
    bool operator==(const ShapeKey &o) const
    {
        return nx == o.nx && ny == o.ny && R == o.R && etl == o.etl && n == o.n && whole == o.whole;
    }
};
constexpr int kShapeMemo = 16;

bool tile_shape(const Geom &g, int n_models, bool whole, TileShape *out)
{
    if (g.model != GBK_MODEL_CUBE || g.u != 1 || g.R > kTileMaxR) return false;
    thread_local ShapeKey keys[kShapeMemo] = {};
    thread_local TileShape shapes[kShapeMemo];
    thread_local int next = 0;
    const ShapeKey key = {g.nx, g.ny, g.R, edge_table_len(g), n_models, whole ? 1 : 0};
    for (int i = 0; i < kShapeMemo; ++i)
        if (keys[i] == key) {
            *out = shapes[i];
            return out->tiles > 0;
        }
    TileShape best = {};
    static const int sizes[] = {1 << 30, 160, 128, 96, 80, 64, 56, 48, 40, 32, 24, 16, 12, 8};
    for (const int bx : sizes) {
        for (const int by : sizes) {
            TileShape s = {};
            const int kx = (g.nx - 1) / bx + 1, ky = (g.ny - 1) / by + 1;  // equal parts of at most that size
            if (whole && (kx > 1 || ky > 1)) continue;
            s.tx = (((g.nx + kx - 1) / kx) + 3) & ~3;
            s.ty = (((g.ny + ky - 1) / ky) + 3) & ~3;
            s.tiles_x = (g.nx + s.tx - 1) / s.tx;
            s.tiles = s.tiles_x * ((g.ny + s.ty - 1) / s.ty);
            s.smem = tile_smem(g, s.tx, s.ty);
            if (s.smem > (size_t)kTileMaxSmem) continue;
            for (int nt = 128; nt <= kTileThreads; nt += 64) {
                const int per_sm = tile_per_sm(s.smem, nt);
                if (per_sm < 1 || (whole && per_sm < 2)) continue;
                s.threads = nt;
                s.cost = tile_cost(g, s, n_models);
                if (best.tiles == 0 || s.cost < best.cost) best = s;
            }
        }
    }
    keys[next] = key;
    shapes[next] = best;
    next = (next + 1) % kShapeMemo;
    *out = best;
    return best.tiles > 0;
}

template <int R, bool MULTI>
static gbk_status launch_rm(const TileArgs &a, const TileShape &ts, cudaStream_t st)
{
    static KernelAttrMemo memo;
    gbk_status s = ensure_kernel_attrs((const void *)tile_kernel<R, MULTI>, ts.smem, false, memo,
                                       "tile evaluator: setting its shared memory");
    if (s) return s;
    const int grid = std::min(a.items, 152 * std::max(1, tile_per_sm(ts.smem, ts.threads)));
    tile_kernel<R, MULTI><<<grid, ts.threads, ts.smem, st>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "tile evaluator launch");
    return GBK_OK;
}

template <int R>
static gbk_status launch_r(const TileArgs &a, const TileShape &ts, cudaStream_t st)
{
    return ts.tiles > 1 ? launch_rm<R, true>(a, ts, st) : launch_rm<R, false>(a, ts, st);
}

gbk_status launch_tile(const Geom &g, const TileShape &ts, int n, const double *params, const gbk_obs *obs,
                       float *maps, double *chi2, float *resid, const TileScratch &scratch, const SplitBatch *batch,
                       int m0, cudaStream_t st)
{
    TileArgs a = {};
    a.g = g;
    a.params = params;
    if (obs) a.obs = *obs;
    a.obs_list = batch ? batch->obs_list : nullptr;
    a.skip = batch ? batch->skip : nullptr;
    a.m0 = m0;
    a.mpg = batch ? batch->mpg : 1;
    a.maps = maps;
    a.chi2 = chi2;
    a.resid = resid;
    a.part = scratch.part;
    a.arrived = scratch.arrived;
    a.tx = ts.tx;
    a.ty = ts.ty;
    a.tiles_x = ts.tiles_x;
    a.tiles = ts.tiles;
    a.items = n * ts.tiles;
    a.vec = g.nx % 2 == 0 && ((uintptr_t)maps % 8) == 0 && ((uintptr_t)resid % 8) == 0;
    switch (g.R) {
    case 0: return launch_r<0>(a, ts, st);
    case 1: return launch_r<1>(a, ts, st);
    case 2: return launch_r<2>(a, ts, st);
    case 3: return launch_r<3>(a, ts, st);
    case 4: return launch_r<4>(a, ts, st);
    case 5: return launch_r<5>(a, ts, st);
    case 6: return launch_r<6>(a, ts, st);
    case 7: return launch_r<7>(a, ts, st);
    case 8: return launch_r<8>(a, ts, st);
    default: return fail(GBK_EUNSUPPORTED, "tile evaluator: PSF radius %d > %d", g.R, kTileMaxR);
    }
}

gbk_status launch_tile_resid_sum(const Geom &g, const TileShape &ts, int n, const double *params, const float *resid,
                                 double *chi2, const TileScratch &scratch, const SplitBatch *batch, int m0,
                                 cudaStream_t st)
{
    ResidSumArgs a = {};
    a.g = g;
    a.params = params;
    a.resid = resid;
    a.skip = batch ? batch->skip : nullptr;
    a.m0 = m0;
    a.mpg = batch ? batch->mpg : 1;
    a.chi2 = chi2;
    a.part = scratch.part;
    a.arrived = scratch.arrived;
    a.tx = ts.tx;
    a.ty = ts.ty;
    a.tiles_x = ts.tiles_x;
    a.tiles = ts.tiles;
    tile_resid_sum_kernel<<<n * ts.tiles, ts.threads, 0, st>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "sum of residuals launch");
    return GBK_OK;
}

// The CTA size for an image held whole, by the CTAs its planes let share an
// SM (24 to 26 warps an SM in each case); 0 where it does not fit.
int tile_ragged_threads(const Geom &g, size_t *smem)
{
    if (g.model != GBK_MODEL_CUBE || g.u != 1 || g.R > kTileMaxR || g.ex > 1024) return 0;
    *smem = tile_smem(g, g.nx, g.ny);
    static const int threads[] = {160, 192, 256, 384, 768};
    for (int i = 0; i < 5; ++i)
        if ((size_t)(5 - i) * (*smem + 3072) <= 227 * 1024) return threads[i];
    return 0;
}

gbk_status launch_tile_ragged(const TileRagged &a, int threads, size_t smem, bool overlap, cudaStream_t st)
{
    static KernelAttrMemo memo;
    gbk_status s = ensure_kernel_attrs((const void *)tile_ragged_kernel, smem, false, memo,
                                       "ragged tile evaluator: setting its shared memory");
    if (s) return s;
    const int per_sm = (int)std::min<size_t>(227 * 1024 / (smem + 3072), 800 / threads);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min(a.items, 152 * std::max(1, per_sm)), 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, tile_ragged_kernel, a);
    if (e != cudaSuccess) return cuda_fail(e, "ragged tile evaluator launch");
    return GBK_OK;
}

}  // namespace gbk
