// k_conv_tma.cu -- the staged separable PSF x LSF convolution (Eq. 9,
// Sec. 2.2.3), built for HBM bandwidth.
//
// One CTA owns a 32 x 32 tile of output spaxels of one model and walks every
// extended channel once:
//   - TMA (cp.async.bulk.tensor, mbarrier completion) loads the tile's input
//     slab of each channel, (32 + 2R) rows x (32 + 2R, rounded to 4) columns,
//     two channels ahead, into a double buffer, so the cube is read from HBM
//     exactly once and the load overlaps the arithmetic;
//   - the x pass gives each thread four adjacent outputs from one float4-
//     loaded row segment (four taps per load); the y pass gives each thread
//     2 x 2 outputs, two columns per packed f32x2 operation;
//   - the z pass keeps, per owned spaxel, the 2 Rz + 1 partial output
//     channels the current input channel contributes to in registers (a
//     shifting window, template-sized), and writes a channel as soon as its
//     window is complete -- coalesced rows of 32 floats.
// Where the tiles alone do not fill the chip the channels are cut as well: a
// CTA walks the extended channels of a range of output channels (the 2 Rz at
// its ends are then read twice).  32 models of 64 x 64 x 128 fine voxels (R =
// 9, Rz = 6) are 128 tiles: 206 us with one CTA each and scalar passes, 160 us
// in halves, 124 us in halves with the passes as above (the whole call: 272 us
// before, 190 us now).  Issue slots bound it: the x pass is scalar, since its
// row pairs would start at odd columns for every other tap.
// Waits on the mbarriers are bounded: a CTA that gives up records a status in
// g_conv_status and stops (the host reports it as GBK_ECUDA via
// gbk_device_status()).
#include <cuda.h>

#include "gbk_api_internal.h"
#include "gbk_internal.cuh"
#include "k_staged.h"
#include "tma_util.cuh"

namespace gbk {

constexpr int kCT = 32;            // output tile edge
constexpr int kCThreads = 256;     // 8 warps
constexpr long kWaitLimit = 1L << 18;  // tries: about one second (3.75 us per failed try_wait)

__device__ int g_conv_status;      // 0 = fine; 1 = a TMA wait timed out

struct ConvTmaArgs {
    Geom g;
    int n_models;
    int tiles_x, tiles_y;
    int box_w;                     // TMA box width, >= 32 + 2R, multiple of 4
    int zparts, zlen;              // ranges of output channels per tile, channels per range
    float *fine;                   // [n][nzf][nyf][nxf]
    size_t f_model_stride;
    int vec2;                      // 1: output rows take 8-byte stores
};

template <int W>
__global__ void __launch_bounds__(kCThreads, (W <= 15 ? 2 : 1)) conv3d_tma_kernel(const __grid_constant__ CUtensorMap tmap,
                                                                 ConvTmaArgs a)
{
    const Geom &g = a.g;
    const int R = g.R, Rz = g.Rz;
    const int SY = kCT + 2 * R, BW = a.box_w;
    const int tiles = a.tiles_x * a.tiles_y;
    const int zpart = blockIdx.x % a.zparts, mt = blockIdx.x / a.zparts;
    const int model = mt / tiles;
    const int t = mt - model * tiles;
    // output channels [k0, k1) come from extended channels [k0, k1 + 2 Rz)
    const int k0 = zpart * a.zlen, k1 = min(g.nzf, k0 + a.zlen);
    const int ne = k1 + 2 * Rz - k0;
    const int ty0 = (t / a.tiles_x) * kCT, tx0 = (t % a.tiles_x) * kCT;
    const int tid = threadIdx.x;

    // A tensor copy's shared-memory destination must be 128-byte aligned: the
    // base is rounded up by hand (the launch adds 128 bytes for that) and each
    // slab is padded to a multiple of 32 floats.
    extern __shared__ __align__(128) float csm_raw[];
    float *csm = csm_raw + (((128u - (smem_u32(csm_raw) & 127u)) & 127u) >> 2);
    const int SS = (SY * BW + 31) & ~31;
    float *slab0 = csm;                        // [SY][BW]
    float *slab1 = slab0 + SS;
    float *X = slab1 + SS;                     // [SY][32] after the x pass
    const int taps = (2 * R + 1 + 3) & ~3;
    float *wxy = X + SY * kCT;                 // 2R+1 taps (padded)
    float *wdup = wxy + taps;                  // the same, each tap twice
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ float s_wz[W];
    __shared__ int s_abort;

    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    // taps (each thread that writes one computes the normalisation itself)
    for (int j = tid; j < taps; j += kCThreads) {
        if (j > 2 * R) {
            wxy[j] = 0.f;
            continue;  // loaded with its group, never used
        }
        float s = 0.f;
        for (int q = -R; q <= R; ++q) s += (R == 0) ? 1.f : gauss_tap(q, g.sig_xy);
        wxy[j] = ((R == 0) ? 1.f : gauss_tap(j - R, g.sig_xy)) / s;
        wdup[2 * j] = wdup[2 * j + 1] = wxy[j];
    }
    if (tid < W) {
        float s = 0.f;
        for (int q = -Rz; q <= Rz; ++q) s += (Rz == 0) ? 1.f : gauss_tap(q, g.sig_z);
        s_wz[tid] = ((Rz == 0) ? 1.f : gauss_tap(tid - Rz, g.sig_z)) / s;
    }
    __syncthreads();

    const uint32_t bytes = (uint32_t)(SY * BW * sizeof(float));
    const int zbase = model * g.ez + k0;
    if (tid == 0) {
        tma_load_slab(&tmap, slab0, &bar[0], tx0, ty0, zbase, bytes);
        if (ne > 1) tma_load_slab(&tmap, slab1, &bar[1], tx0, ty0, zbase + 1, bytes);
    }
    f32x2 wz[W];
#pragma unroll
    for (int q = 0; q < W; ++q) wz[q] = pk2(s_wz[q], s_wz[q]);

    // y-pass / z-pass ownership: columns 2 c, 2 c + 1 (packed pairs), rows 2 gq, 2 gq + 1
    const int c = tid & 15, gq = tid >> 4;
    f32x2 acc[2][W];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < W; ++q) acc[p][q] = pk2(0.f, 0.f);
    float *F = a.fine + (size_t)model * a.f_model_stride;
    const size_t fplane = (size_t)g.nyf * g.nxf;
    const int ox = tx0 + 2 * c;
    const int nitems = SY * (kCT / 4);  // x pass: (row, 4-column group)

    for (int e = 0; e < ne; ++e) {  // extended channel k0 + e
        float *slab = (e & 1) ? slab1 : slab0;
        if (!mbar_wait(&bar[e & 1], (uint32_t)((e >> 1) & 1), kWaitLimit)) {
            if (atomicExch(&s_abort, 1) == 0) atomicExch(&g_conv_status, 1);
        }
        __syncthreads();
        if (s_abort) {
            // give the other buffer's copy, if one is in flight, a bounded
            // chance to land before the CTA leaves
            if (tid == 0 && e + 1 < ne) mbar_wait(&bar[(e + 1) & 1], (uint32_t)(((e + 1) >> 1) & 1), kWaitLimit);
            return;  // every thread sees the same flag after the barrier
        }
        // x pass: X[r][4 m .. 4 m + 3] from slab[r][4 m .. 4 m + 3 + 2R]
        for (int it = tid; it < nitems; it += kCThreads) {
            int r = it >> 3, m = it & 7;
            const float4 *row = reinterpret_cast<const float4 *>(slab + r * BW + 4 * m);
            float o0 = 0.f, o1 = 0.f, o2 = 0.f, o3 = 0.f;
            float4 p = row[0];
            int j = 0;
#pragma unroll 2
            for (; j + 3 <= 2 * R; j += 4) {  // four taps per 16-byte load
                const float4 n = row[j / 4 + 1], w = *reinterpret_cast<const float4 *>(wxy + j);
                o0 = fmaf(w.x, p.x, o0); o1 = fmaf(w.x, p.y, o1); o2 = fmaf(w.x, p.z, o2); o3 = fmaf(w.x, p.w, o3);
                o0 = fmaf(w.y, p.y, o0); o1 = fmaf(w.y, p.z, o1); o2 = fmaf(w.y, p.w, o2); o3 = fmaf(w.y, n.x, o3);
                o0 = fmaf(w.z, p.z, o0); o1 = fmaf(w.z, p.w, o1); o2 = fmaf(w.z, n.x, o2); o3 = fmaf(w.z, n.y, o3);
                o0 = fmaf(w.w, p.w, o0); o1 = fmaf(w.w, n.x, o1); o2 = fmaf(w.w, n.y, o2); o3 = fmaf(w.w, n.z, o3);
                p = n;
            }
            {  // one tap (R even) or three (R odd) are left; BW is a multiple of 4, so the row holds n
                const float4 w = *reinterpret_cast<const float4 *>(wxy + j);
                o0 = fmaf(w.x, p.x, o0); o1 = fmaf(w.x, p.y, o1); o2 = fmaf(w.x, p.z, o2); o3 = fmaf(w.x, p.w, o3);
                if (R & 1) {
                    const float4 n = row[j / 4 + 1];
                    o0 = fmaf(w.y, p.y, o0); o1 = fmaf(w.y, p.z, o1); o2 = fmaf(w.y, p.w, o2); o3 = fmaf(w.y, n.x, o3);
                    o0 = fmaf(w.z, p.z, o0); o1 = fmaf(w.z, p.w, o1); o2 = fmaf(w.z, n.x, o2); o3 = fmaf(w.z, n.y, o3);
                }
            }
            *reinterpret_cast<float4 *>(X + r * kCT + 4 * m) = make_float4(o0, o1, o2, o3);
        }
        __syncthreads();
        // the slab is consumed: refill it with channel e + 2
        if (tid == 0 && e + 2 < ne) tma_load_slab(&tmap, slab, &bar[e & 1], tx0, ty0, zbase + e + 2, bytes);
        // y pass: rows 2 gq, 2 gq + 1 of columns 2 c, 2 c + 1
        f32x2 yv[2] = {pk2(0.f, 0.f), pk2(0.f, 0.f)};
        {
            const f32x2 *col = reinterpret_cast<const f32x2 *>(X + 2 * gq * kCT + 2 * c);
            const f32x2 *w2 = reinterpret_cast<const f32x2 *>(wdup);
            f32x2 v0 = col[0];
#pragma unroll 4
            for (int j = 0; j <= 2 * R; ++j) {
                const f32x2 v1 = col[(j + 1) * (kCT / 2)];
                yv[0] = fma2(w2[j], v0, yv[0]);
                yv[1] = fma2(w2[j], v1, yv[1]);
                v0 = v1;
            }
        }
        // z pass: slot q holds output channel e - 2 Rz + q, weight wz[q]; the
        // sums move down one slot as they take the channel
        const int k = k0 + e - 2 * Rz;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const f32x2 out = fma2(wz[0], yv[p], acc[p][0]);
#pragma unroll
            for (int q = 1; q < W; ++q) acc[p][q - 1] = fma2(wz[q], yv[p], acc[p][q]);
            const int oy = ty0 + 2 * gq + p;
            if (k >= k0 && ox < g.nxf && oy < g.nyf) {
                float *dst = F + (size_t)k * fplane + (size_t)oy * g.nxf + ox;
                if (a.vec2) {
                    *reinterpret_cast<f32x2 *>(dst) = out;
                } else {
                    float lo, hi;
                    upk2(out, lo, hi);
                    dst[0] = lo;
                    if (ox + 1 < g.nxf) dst[1] = hi;
                }
            }
        }
        // X is rewritten by the next x pass
        __syncthreads();
    }
}

// ----------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

size_t conv_tma_smem_bytes(const Geom &g)
{
    int SY = kCT + 2 * g.R, BW = (kCT + 2 * g.R + 3) & ~3;
    int SS = (SY * BW + 31) & ~31;
    return 128 + sizeof(float) * (size_t)(2 * SS + SY * kCT + 3 * ((2 * g.R + 1 + 3) & ~3));
}

bool conv_tma_supported(const Geom &g)
{
    int W = 2 * g.Rz + 1;
    return W <= 23 && (kCT + 2 * g.R) <= 256 && conv_tma_smem_bytes(g) <= 200 * 1024 + 8 * (size_t)((2 * g.R + 1 + 3) & ~3) && encode_fn() != nullptr;
}

template <int W>
static gbk_status launch_w(const CUtensorMap &tm, const ConvTmaArgs &a, size_t smem, int blocks, cudaStream_t st)
{
    static KernelAttrMemo memo;
    gbk_status s = ensure_kernel_attrs((const void *)conv3d_tma_kernel<W>, smem, false, memo,
                                       "TMA convolution: setting dynamic shared memory");
    if (s) return s;
    conv3d_tma_kernel<W><<<blocks, kCThreads, smem, st>>>(tm, a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "TMA convolution launch");
    return GBK_OK;
}

gbk_status launch_conv_tma(const StagedArgs &sa, cudaStream_t st)
{
    const Geom &g = sa.g;
    EncodeTiledFn enc = encode_fn();
    if (!enc) return fail(GBK_EUNSUPPORTED, "cuTensorMapEncodeTiled is not available from the driver");
    ConvTmaArgs a = {};
    a.g = g;
    a.n_models = sa.n_models;
    a.tiles_x = (g.nxf + kCT - 1) / kCT;
    a.tiles_y = (g.nyf + kCT - 1) / kCT;
    a.box_w = (kCT + 2 * g.R + 3) & ~3;
    a.fine = sa.fine;
    a.f_model_stride = sa.f_model_stride;
    a.vec2 = g.nxf % 2 == 0 && sa.f_model_stride % 2 == 0 && reinterpret_cast<uintptr_t>(sa.fine) % 8 == 0;
    CUtensorMap tm;
    cuuint64_t dims[3] = {(cuuint64_t)sa.e_pitch, (cuuint64_t)g.ey, (cuuint64_t)g.ez * (cuuint64_t)sa.n_models};
    cuuint64_t strides[2] = {(cuuint64_t)sa.e_pitch * sizeof(float), (cuuint64_t)sa.e_pitch * g.ey * sizeof(float)};
    cuuint32_t box[3] = {(cuuint32_t)a.box_w, (cuuint32_t)(kCT + 2 * g.R), 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(&tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, (void *)sa.ext, dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(GBK_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    size_t smem = conv_tma_smem_bytes(g);
    // ranges of channels: the count with the shortest queue of whole walks
    const long tiles = (long)a.tiles_x * a.tiles_y * sa.n_models;
    const long slots = 152 * (2 * g.Rz + 1 <= 15 && 2 * (smem + 1024) <= 228 * 1024 ? 2 : 1);
    long best = 0;
    a.zparts = 1;
    a.zlen = g.nzf;
    for (int z = 1; z <= 8 && z <= g.nzf; ++z) {
        const int len = (g.nzf + z - 1) / z;
        const long cost = ((tiles * z + slots - 1) / slots) * (len + 2 * g.Rz);
        if (z == 1 || cost * 10 < best * 9) {  // a tenth better, for the channels read twice
            best = cost;
            a.zparts = (g.nzf + len - 1) / len;
            a.zlen = len;
        }
    }
    int blocks = (int)(tiles * a.zparts);
    switch (2 * g.Rz + 1) {
    case 1: return launch_w<1>(tm, a, smem, blocks, st);
    case 3: return launch_w<3>(tm, a, smem, blocks, st);
    case 5: return launch_w<5>(tm, a, smem, blocks, st);
    case 7: return launch_w<7>(tm, a, smem, blocks, st);
    case 9: return launch_w<9>(tm, a, smem, blocks, st);
    case 11: return launch_w<11>(tm, a, smem, blocks, st);
    case 13: return launch_w<13>(tm, a, smem, blocks, st);
    case 15: return launch_w<15>(tm, a, smem, blocks, st);
    case 17: return launch_w<17>(tm, a, smem, blocks, st);
    case 19: return launch_w<19>(tm, a, smem, blocks, st);
    case 21: return launch_w<21>(tm, a, smem, blocks, st);
    case 23: return launch_w<23>(tm, a, smem, blocks, st);
    default: return fail(GBK_EUNSUPPORTED, "LSF window %d not served by the TMA convolution", 2 * g.Rz + 1);
    }
}

gbk_status conv_status_read(int *v)
{
    int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(v, g_conv_status, sizeof(int));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_conv_status, &zero, sizeof(int));
    if (e != cudaSuccess) return cuda_fail(e, "reading the convolution status");
    return GBK_OK;
}

}  // namespace gbk
