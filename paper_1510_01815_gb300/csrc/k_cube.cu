// k_cube.cu -- convolved model cubes and their moments in one kernel (u = 1,
// PSF radii up to 8, LSF radii up to 6): the model cube never goes to memory.
//
// The staged chain writes the extended model cube, reads it for the
// convolution, writes the data cube and reads it again for the moments: four
// passes over HBM, of which a caller needs one (the data cube).  Here one CTA
// of 256 threads owns a 64 x 16 tile of output spaxels of one model and walks
// the channels in batches of NC = 256 / (32 + R) (R even):
//   - the tile's line velocities and amplitudes, with the halo, are computed
//     once and stay in shared memory;
//   - pass 1 (line and PSF along y): a thread takes one channel and one column
//     pair, evaluates the line at each row (one ex2 per voxel) and adds it to
//     the 2 R + 1 rows that it feeds, all in registers.  A batch of channels
//     gives every thread a task (a single channel has 32 + R);
//   - pass 2 (PSF along x): a thread owns four adjacent spaxels of one row,
//     one 16-byte load per four taps;
//   - pass 3 (LSF along z): a transposed FIR in registers, then the stores
//     and the moment sums about the spaxel's own (clamped) line velocity.
// One barrier per batch; the rows between passes 1 and 2 are double-buffered.
// One instance per PSF radius; LSF radii are rounded up to even numbers.
// Terms and their order are those of the staged chain (y, x, z, moments by
// channel), and so are the bits.
//
// Where the tiles do not fill the chip the channels are cut into ranges
// (zparts), whose moments then take moments_kernel's pass over the cube.
//
// 256 models of 64 x 64 x 64 (R = 5, Rz = 3): 284 us by the staged chain (1.3
// GB moved), 176 us here (268 MB).
// The packed FMAs (two passes of the FMA pipe each, busy 60 %) and their issue
// slots (63 %) bound it; 31 models of 142 x 128 x 102: 256 -> 159 us, 4 models
// of 64 x 25 x 74: 62 -> 23 us.
#include <cmath>
#include <cstring>

#include "gbk_api_internal.h"
#include "gbk_internal.cuh"
#include "k_staged.h"

namespace gbk {

constexpr int kQX = 64, kQY = 16;  // output tile
constexpr int kQThreads = 256;
constexpr int kQRmax = 8;          // largest PSF radius served
// Largest LSF radius served: radii 7 and 8 hold 64 registers of partial sums,
// one CTA per SM instead of two, and the staged chain is the faster one (one
// cube of a call took 117 us against 54 us).
constexpr int kQRzMax = 6;

struct CubeArgs {
    Geom g;
    const double *params;
    float *cubes;                // [n][nz][ny][nx]
    float *maps;                 // [n][3][ny][nx] or null (null when zparts > 1)
    int tiles_x, tiles;          // tiles per row, per model
    int zparts, zlen;            // ranges of output channels per tile, channels per range
    f32x2 w2[2 * kQRmax + 1];    // PSF taps (w, w), normalised, centred in 2 R + 1
    f32x2 wz2[2 * kQRzMax + 1];  // LSF taps
};

template <int R>
struct CubeDims {
    static constexpr int H = (R + 1) & ~1;       // halo: even, so that rows start on 16 bytes
    static constexpr int O = H - R;              // first halo row and column in use
    static constexpr int CW = kQX + 2 * H;       // columns with the halo
    static constexpr int CP = CW / 2;            // ... as pairs
    static constexpr int SY = kQY + 2 * H;       // rows with the halo
    static constexpr int NC = kQThreads / CP;    // channels per batch
    static constexpr int YF = NC * kQY * CW;     // floats per row buffer
    static constexpr size_t smem = sizeof(float) * ((size_t)4 * SY * CP + 2 * YF);
};

template <int R, int RZ>
__global__ void __launch_bounds__(kQThreads, 2) cube_kernel(const __grid_constant__ CubeArgs a)
{
    using D = CubeDims<R>;
    const Geom &g = a.g;
    const int zpart = blockIdx.x % a.zparts, mt = blockIdx.x / a.zparts;
    const int model = mt / a.tiles, t = mt - model * a.tiles;
    const int ty0 = (t / a.tiles_x) * kQY, tx0 = (t % a.tiles_x) * kQX;
    const int k0 = zpart * a.zlen, k1 = min(g.nz, k0 + a.zlen);
    const int ne = k1 - k0 + 2 * RZ;  // channels k0 - RZ .. k1 + RZ - 1
    const int tid = threadIdx.x;

    extern __shared__ __align__(16) float qsm[];
    float4 *const tab = reinterpret_cast<float4 *>(qsm);  // [SY][CP]: (-v, -v', A, A') of a column pair
    float *const Y = qsm + 4 * D::SY * D::CP;              // [2][NC][16][CW]
    __shared__ ModelConst mc;
    if (tid == 0) mc = model_const(a.params + (size_t)model * GBK_NPAR, g);
    __syncthreads();
    const float al = mc.alpha;
    for (int i = tid; i < D::SY * D::CW; i += kQThreads) {
        const int r = i / D::CW, col = i - r * D::CW;
        const float2 vb = line_at(mc, (float)(tx0 + col - D::H), (float)(ty0 + r - D::H));
        float *e = qsm + 4 * (r * D::CP + (col >> 1)) + (col & 1);
        e[0] = -vb.x;
        e[2] = mc.valid ? mc.amp * vb.y : __int_as_float(0x7fc00000);
    }
    __syncthreads();

    // pass 1: channel ch of the batch, columns 2 cq, 2 cq + 1
    const int ch = tid / D::CP, cq = tid - ch * D::CP;
    // passes 2 and 3: spaxels ox .. ox + 3 of row oy
    const int row = tid >> 4, c4 = tid & 15;
    const int ox = tx0 + 4 * c4, oy = ty0 + row;
    const size_t np = (size_t)g.nx * g.ny;
    const bool vec = (g.nx & 3) == 0;
    float *F = a.cubes + ((size_t)model * g.nz + k0) * np + (size_t)oy * g.nx + ox;
    const f32x2 Z = pk2(0.f, 0.f), AL = pk2(al, al), DV = pk2(g.dv, g.dv);
    f32x2 P[2][2 * RZ];  // partial sums of the output channels in progress
#pragma unroll
    for (int d = 0; d < 2 * RZ; ++d) P[0][d] = P[1][d] = Z;
    f32x2 base[2], S0[2] = {Z, Z}, S1[2] = {Z, Z}, S2[2] = {Z, Z};  // moment sums of the four spaxels
    float cen[4];
    if (a.maps) {
        float b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 cb = moment_centre(mc, g, (float)(ox + q), (float)oy);
            cen[q] = cb.x;
            b[q] = cb.y;
        }
        base[0] = pk2(b[0], b[1]);
        base[1] = pk2(b[2], b[3]);
    }

    int buf = 0;
    for (int e0 = 0; e0 < ne; e0 += D::NC, buf ^= 1) {
        float *const Yb = Y + buf * D::YF;
        // ---- pass 1: the line at each row of a column pair, and the PSF along y ----
        if (ch < D::NC && e0 + ch < ne) {
            const float v = g.vc + ((float)(k0 + e0 + ch - RZ) - 0.5f * (float)(g.nz - 1)) * g.dv;
            const f32x2 V = pk2(v, v);
            const float4 *src = tab + cq;
            float *dst = Yb + ch * kQY * D::CW + 2 * cq;
            f32x2 acc[2 * R + 1];
#pragma unroll
            for (int i = 0; i < kQY + 2 * R; ++i) {
                const float4 s = src[(i + D::O) * D::CP];
                const f32x2 u = mul2(AL, add2(V, pk2(s.x, s.y)));
                float w0, w1;
                upk2(mul2(u, u), w0, w1);
                const f32x2 x = mul2(pk2(s.z, s.w), pk2(ex2_approx(-w0), ex2_approx(-w1)));
#pragma unroll
                for (int d = 0; d <= 2 * R; ++d) {  // output row r takes this row with tap d
                    const int r = i - d;
                    if (r < 0 || r >= kQY) continue;
                    f32x2 &o = acc[r % (2 * R + 1)];
                    o = d ? fma2(a.w2[d], x, o) : mul2(a.w2[0], x);
                    if (d == 2 * R) *reinterpret_cast<f32x2 *>(dst + r * D::CW) = o;
                }
            }
        }
        __syncthreads();
        // ---- passes 2 and 3, channel by channel ----
#pragma unroll 1
        for (int q = 0; q < D::NC && e0 + q < ne; ++q) {
            const float4 *yr = reinterpret_cast<const float4 *>(Yb + (q * kQY + row) * D::CW) + c4;
            float f[4 + 2 * D::H];
#pragma unroll
            for (int m = 0; m <= D::H / 2; ++m) {
                const float4 x = yr[m];
                f[4 * m] = x.x; f[4 * m + 1] = x.y; f[4 * m + 2] = x.z; f[4 * m + 3] = x.w;
            }
            f32x2 v[2] = {Z, Z};
#pragma unroll
            for (int j = 0; j <= 2 * R; ++j) {
                v[0] = fma2(a.w2[j], pk2(f[D::O + j], f[D::O + j + 1]), v[0]);
                v[1] = fma2(a.w2[j], pk2(f[D::O + j + 2], f[D::O + j + 3]), v[1]);
            }
            f32x2 o[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                o[h] = fma2(a.wz2[2 * RZ], v[h], P[h][0]);
#pragma unroll
                for (int d = 1; d < 2 * RZ; ++d) P[h][d - 1] = fma2(a.wz2[2 * RZ - d], v[h], P[h][d]);
                P[h][2 * RZ - 1] = mul2(a.wz2[0], v[h]);
            }
            const int k = e0 + q - 2 * RZ;  // the range's channel that is complete
            if (k < 0) continue;
            float4 out;
            upk2(o[0], out.x, out.y);
            upk2(o[1], out.z, out.w);
            if (oy < g.ny) {
                if (vec) {
                    if (ox < g.nx) *reinterpret_cast<float4 *>(F) = out;
                } else {
                    if (ox < g.nx) F[0] = out.x;
                    if (ox + 1 < g.nx) F[1] = out.y;
                    if (ox + 2 < g.nx) F[2] = out.z;
                    if (ox + 3 < g.nx) F[3] = out.w;
                }
            }
            F += np;
            if (!a.maps) continue;
            const float fk = (float)k;  // k0 = 0 where the moments are taken
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const f32x2 dd = fma2(pk2(fk, fk), DV, base[h]);
                const f32x2 tt = mul2(o[h], dd);
                S0[h] = add2(S0[h], o[h]);
                S1[h] = fma2(o[h], dd, S1[h]);
                S2[h] = fma2(tt, dd, S2[h]);
            }
        }
    }
    if (!a.maps || oy >= g.ny) return;
    float *mp = a.maps + (size_t)model * 3 * np + (size_t)oy * g.nx + ox;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (ox + q >= g.nx) break;
        float s[3][2], m0, m1, m2;
        bool valid;
        upk2(S0[q >> 1], s[0][0], s[0][1]);
        upk2(S1[q >> 1], s[1][0], s[1][1]);
        upk2(S2[q >> 1], s[2][0], s[2][1]);
        finish_moments(s[0][q & 1], s[1][q & 1], s[2][q & 1], cen[q], mc, m0, m1, m2, valid);
        mp[q] = m0;
        mp[np + q] = m1;
        mp[2 * np + q] = m2;
    }
}

template <int R, int RZ>
static gbk_status launch_rr(const CubeArgs &a, long blocks, cudaStream_t st)
{
    static KernelAttrMemo memo;
    const size_t smem = CubeDims<R>::smem;
    gbk_status s = ensure_kernel_attrs((const void *)cube_kernel<R, RZ>, smem, false, memo,
                                       "model cube: setting dynamic shared memory");
    if (s) return s;
    cube_kernel<R, RZ><<<(unsigned)blocks, kQThreads, smem, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "model cube launch");
    return GBK_OK;
}

template <int R>
static gbk_status launch_r(int rz, const CubeArgs &a, long blocks, cudaStream_t st)
{
    switch (rz) {
    case 2: return launch_rr<R, 2>(a, blocks, st);
    case 4: return launch_rr<R, 4>(a, blocks, st);
    default: return launch_rr<R, 6>(a, blocks, st);
    }
}

bool cube_supported(const Geom &g, int n_models)
{
    const long tiles = (long)((g.nx + kQX - 1) / kQX) * ((g.ny + kQY - 1) / kQY);
    return g.model == GBK_MODEL_CUBE && g.u == 1 && g.R <= kQRmax && g.Rz <= kQRzMax &&
           tiles * n_models <= 0x7fffffffL / 8;  // eight ranges at most
}

gbk_status launch_cube(const Geom &g, int n_models, const double *params, float *cubes, float *maps, cudaStream_t st,
                       bool *moments_left)
{
    CubeArgs a = {};
    a.g = g;
    a.params = params;
    a.cubes = cubes;
    // instances: PSF radii 1 .. 8, LSF radii 2, 4, 6 (taps 0 outside the true radius)
    const int R = g.R < 1 ? 1 : g.R, RZ = g.Rz < 2 ? 2 : (g.Rz + 1) & ~1;
    // normalised Gaussian taps of radius `rt`, centred in a window of radius `ri`
    auto taps = [](int rt, int ri, float sigma, f32x2 *out) {
        double w[2 * kQRmax + 1], sum = 0.0;
        for (int j = -rt; j <= rt; ++j) {
            const double t = (rt == 0) ? 0.0 : (double)j / (double)sigma;
            w[j + rt] = std::exp(-0.5 * t * t);
            sum += w[j + rt];
        }
        for (int j = -rt; j <= rt; ++j) {
            const float f = (float)(w[j + rt] / sum);
            uint32_t b;
            std::memcpy(&b, &f, 4);
            out[j + ri] = ((f32x2)b << 32) | (f32x2)b;
        }
    };
    taps(g.R, R, g.sig_xy, a.w2);
    taps(g.Rz, RZ, g.sig_z, a.wz2);
    a.tiles_x = (g.nx + kQX - 1) / kQX;
    a.tiles = a.tiles_x * ((g.ny + kQY - 1) / kQY);
    // Ranges of channels: a cut costs 2 RZ channels more per range and, for
    // the maps, another pass over the cube, so it has to shorten the queue by
    // a quarter (in practice: batches of less than one wave).
    const long slots = 152 * 2, tiles = (long)a.tiles * n_models;
    long best = 0;
    a.zparts = 1;
    a.zlen = g.nz;
    for (int z = 1; z <= 8 && z <= g.nz; ++z) {
        const int len = (g.nz + z - 1) / z;
        const long cost = ((tiles * z + slots - 1) / slots) * (len + 2 * RZ);
        if (z == 1 || cost * 4 < best * 3) {
            best = cost;
            a.zparts = (g.nz + len - 1) / len;
            a.zlen = len;
        }
    }
    a.maps = a.zparts == 1 ? maps : nullptr;
    *moments_left = maps && a.zparts > 1;
    const long blocks = tiles * a.zparts;
    switch (R) {
    case 1: return launch_r<1>(RZ, a, blocks, st);
    case 2: return launch_r<2>(RZ, a, blocks, st);
    case 3: return launch_r<3>(RZ, a, blocks, st);
    case 4: return launch_r<4>(RZ, a, blocks, st);
    case 5: return launch_r<5>(RZ, a, blocks, st);
    case 6: return launch_r<6>(RZ, a, blocks, st);
    case 7: return launch_r<7>(RZ, a, blocks, st);
    default: return launch_r<8>(RZ, a, blocks, st);
    }
}

}  // namespace gbk
