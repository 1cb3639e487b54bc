// k_staged.h -- launchers of the staged (cube-materialising) kernels.
#pragma once

#include "gbk_internal.cuh"

namespace gbk {

constexpr int kConvTX = 32;
constexpr int kConvTY = 8;

struct StagedArgs {
    Geom g;
    int n_models;
    const double *params;    // [n][GBK_NPAR]
    float *ext;              // fine extended model cube, [n][ez][ey][e_pitch]
    int e_pitch;             // row pitch of ext in floats (multiple of 4, >= ex)
    size_t e_model_stride;   // floats per model in ext
    float *fine;             // convolved fine cube [n][nzf][nyf][nxf]
    size_t f_model_stride;
    float *data;             // data-resolution cube [n][nz][ny][nx] (== fine when u == 1)
    size_t d_model_stride;
    float *maps;             // [n][3][ny][nx] or null
    double *chi2;            // [n] or null
    float *resid;            // [n][2][ny][nx] or null
    double *partials;        // [n][ceil(nx*ny/256)] when chi2 is set
    gbk_obs obs;
};

// Line-of-sight velocity (Eq. 8; Vrot(r) cos(theta) as [Vrot(r) / r] x_e, Eqs.
// 4 and 6, whose r -> 0 limit is (2/pi) Vmax / r_t) and surface brightness (Eq.
// 5) at sky position (x, y) in data pixels, every rounding spelt out: the
// staged chain and the one-kernel cubes get the same bits whatever the
// compiler would contract around the call (a call that is not inlined does that too, at 2 % of the chain's time).
static __device__ __forceinline__ float2 line_at(const ModelConst &c, float x, float y)
{
    const float dx = __fsub_rn(x, c.x0), dy = __fsub_rn(y, c.y0);
    const float xe = __fmaf_rn(dy, c.cos_pa, -__fmul_rn(dx, c.sin_pa));
    const float ye = __fmaf_rn(-dx, c.cos_pa, -__fmul_rn(dy, c.sin_pa));
    const float yd = __fmul_rn(ye, c.inv_cos_i);
    const float r = sqrtf(__fmaf_rn(xe, xe, __fmul_rn(yd, yd)));
    const float f = (r > 0.f) ? __fdiv_rn(__fmul_rn(c.vrot_k, atanf(__fmul_rn(r, c.inv_rt))), r)
                              : __fmul_rn(c.vrot_k, c.inv_rt);
    return make_float2(__fmaf_rn(__fmul_rn(f, xe), c.sin_i, c.vsys),
                       __fmul_rn(c.i0, expf(-__fmul_rn(r, c.inv_h))));
}

// Centre of a spaxel's moment sums -- v_los clamped into the band -- and the
// velocity of channel 0 about it (roundings spelt out, as above).
static __device__ __forceinline__ float2 moment_centre(const ModelConst &c, const Geom &g, float x, float y)
{
    const float half = 0.5f * (float)(g.nz - 1);
    const float v_lo = __fmaf_rn(-half, g.dv, g.vc), v_hi = __fmaf_rn(half, g.dv, g.vc);
    const float cen = fminf(fmaxf(line_at(c, x, y).x, v_lo), v_hi);
    return make_float2(cen, __fsub_rn(v_lo, cen));
}

// Map values of a spaxel from its moment sums about `cen`.
__device__ __forceinline__ void finish_moments(float s0, float s1, float s2, float cen,
                                               const ModelConst &c, float &m0, float &m1, float &m2,
                                               bool &valid)
{
    valid = s0 > kInvalidFraction * c.i0;
    if (!c.valid) {
        m0 = m1 = m2 = __int_as_float(0x7fc00000);
    } else if (valid) {
        float mu = s1 / s0;
        m0 = s0;
        m1 = cen + mu;
        m2 = sqrtf(fmaxf(fmaf(-mu, mu, s2 / s0), 0.f));
    } else {
        m0 = 0.f; m1 = c.vsys; m2 = 0.f;
    }
}

size_t conv_smem_bytes(const Geom &g);
bool conv_tma_supported(const Geom &g);
gbk_status launch_conv_tma(const StagedArgs &a, cudaStream_t stream);
// ev (optional): five events recorded at the stage boundaries -- before the
// model cube, after it, after the convolution, after the down-sampling and
// after the moments and chi2.
gbk_status launch_staged(const StagedArgs &a, bool want_moments, cudaStream_t stream,
                         cudaEvent_t *ev = nullptr);
cudaError_t launch_chi2_maps(int nx, int ny, int n_models, const float *maps, const gbk_obs &obs,
                             double *chi2, float *resid, cudaStream_t stream);

gbk_status conv_status_read(int *v);
// Register-FIR convolution for PSF and LSF radii up to 8 (k_conv_fir.cu).
bool conv_fir_supported(const Geom &g);
gbk_status launch_conv_fir(const StagedArgs &a, cudaStream_t stream);
gbk_status conv_fir_status_read(int *v);
// Cubes (and maps) of u = 1 models with small radii, the model cube kept on
// chip (k_cube.cu).  *moments_left: the maps are still to be taken from the
// cubes (launch_moments).
bool cube_supported(const Geom &g, int n_models);
gbk_status launch_cube(const Geom &g, int n_models, const double *params, float *cubes, float *maps, cudaStream_t st,
                       bool *moments_left);
gbk_status launch_moments(const StagedArgs &a, cudaStream_t stream);

}  // namespace gbk
