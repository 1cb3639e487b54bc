// k_split.cu -- host side of the split path (GBK_PATH_SPLIT): its workspace
// and the calls of the one-kernel evaluator (k_tile.cu) that serve it.  Also
// what the two-stage Jacobian (k_tsplit.cu) shares with it: the driver's
// tensor-map encoder and the auxiliary stream.
//
// The path's first form ran two kernels a chunk of models, the lines with the
// PSF along x and the PSF along y with the moments, meeting in an L2-resident
// buffer.  Once the lines cost a few dozen operations a spaxel instead of a
// channel loop, that buffer, its halo and the launches were most of the time:
// 400 Fabry-Perot models (192 x 192 x 48) take 0.51 ms with the sampled lines
// in two stages, 0.33 ms with the closed-form lines in two stages and 0.28 ms
// in one kernel; 2048 models of 32 x 32 x 64 take 0.100, 0.078 and 0.049 ms.
#include <algorithm>
#include <mutex>

#include "fused_line.cuh"
#include "gbk_api_internal.h"
#include "k_split.h"
#include "k_tile.h"

namespace gbk {

constexpr size_t kSplitL2Budget = (size_t)48 << 20;  // a chunk's share of the workspace
constexpr int kSplitMaxEx = 1024;                    // widest extended row served
constexpr int kSplitTX = 64, kSplitTY = 32;          // tiles the workspace formula counts

SplitEncodeFn split_encode_fn()
{
    static SplitEncodeFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, []() {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (SplitEncodeFn)p;
    });
    return fn;
}

// The workspace: a region whose size is part of the interface (callers keep
// sizes between calls), of which the evaluator uses the planes' part for the
// chi2 parts and arrival counters of images cut into tiles.
struct SplitLayout {
    size_t pl_off, pl_bytes, total;
};

static size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

static SplitLayout split_layout(const Geom &g, int n_models)
{
    SplitLayout L = {};
    const int nxp = (g.nx + 3) & ~3;
    const size_t plb = (size_t)4 * g.ey * nxp * sizeof(float);
    size_t chunk = kSplitL2Budget / plb;
    if (chunk < 1) chunk = 1;
    if (chunk > (size_t)n_models) chunk = (size_t)n_models;
    const size_t nchunks = ((size_t)n_models + chunk - 1) / chunk;
    chunk = ((size_t)n_models + nchunks - 1) / nchunks;  // balanced chunks
    const size_t nbuf = (size_t)n_models > chunk ? 2 : 1;
    const size_t tiles = (size_t)((g.nx + kSplitTX - 1) / kSplitTX) * ((g.ny + kSplitTY - 1) / kSplitTY);
    const size_t tab = 2 * kSplitMaxR + 8 + 3 * edge_table_len(g);
    L.pl_off = al256((size_t)n_models * sizeof(ModelConst)) + al256(tab * sizeof(float));
    L.pl_bytes = nbuf * chunk * plb;
    L.total = L.pl_off + al256(L.pl_bytes) + al256(chunk * tiles * sizeof(double)) + al256(chunk * sizeof(unsigned));
    return L;
}

bool split_supported(const Geom &g)
{
    TileShape ts;
    return g.model == GBK_MODEL_CUBE && g.u == 1 && g.R <= kSplitMaxR && g.ex <= kSplitMaxEx &&
           (size_t)(4 * (((g.ex + 3) & ~3) + 4) + 3 * edge_table_len(g)) * sizeof(float) <= 200 * 1024 &&
           tile_shape(g, 1, false, &ts);
}

size_t split_workspace_bytes(const Geom &g, int n_models)
{
    if (!split_supported(g) || n_models < 1) return 0;
    return split_layout(g, n_models).total;
}

gbk_status split_aux(SplitAux **out)
{
    constexpr int kMaxDev = 64;
    thread_local SplitAux aux[kMaxDev];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "split evaluator: current device");
    if (dev < 0 || dev >= kMaxDev) return fail(GBK_EUNSUPPORTED, "split evaluator: device ordinal %d", dev);
    SplitAux &x = aux[dev];
    if (!x.s) {
        SplitAux y;
        if ((e = cudaStreamCreateWithFlags(&y.s, cudaStreamNonBlocking)) ||
            (e = cudaEventCreateWithFlags(&y.line[0], cudaEventDisableTiming)) ||
            (e = cudaEventCreateWithFlags(&y.line[1], cudaEventDisableTiming)) ||
            (e = cudaEventCreateWithFlags(&y.psf[0], cudaEventDisableTiming)) ||
            (e = cudaEventCreateWithFlags(&y.psf[1], cudaEventDisableTiming)) ||
            (e = cudaEventCreateWithFlags(&y.start, cudaEventDisableTiming)) ||
            (e = cudaEventCreateWithFlags(&y.obs, cudaEventDisableTiming)))
            return cuda_fail(e, "split evaluator: creating the PSF stages' stream");
        x = y;
    }
    *out = &x;
    return GBK_OK;
}

gbk_status launch_split(const Geom &g, int n, const double *params, const gbk_obs *obs, float *maps, double *chi2,
                        float *resid, void *ws, size_t ws_bytes, cudaStream_t st, SplitTimer *timer,
                        const SplitBatch *batch, cudaEvent_t obs_ready)
{
    if (batch && batch->mpg < 1) return fail(GBK_EINVAL, "split evaluator: models per galaxy must be >= 1");
    if ((chi2 || resid) && !obs && !(batch && batch->obs_list))
        return fail(GBK_EINVAL, "split evaluator: chi2 and residuals need observed maps");
    TileShape ts;
    if (!split_supported(g) || !tile_shape(g, chi2 ? kTileChi2Batch : n, false, &ts))
        return fail(GBK_EUNSUPPORTED, "the split evaluator does not serve this geometry");
    if (n == 0) return GBK_OK;
    const SplitLayout L = split_layout(g, n);
    if (!ws || ws_bytes < L.total)
        return fail(GBK_EWORKSPACE, "the split evaluator needs %zu bytes of workspace (got %zu)", L.total, ws_bytes);
    cudaError_t e;
    if (obs_ready && (e = cudaStreamWaitEvent(st, obs_ready, 0)) != cudaSuccess)
        return cuda_fail(e, "split evaluator: waiting for the observed maps");
    // models per launch: as many as the chi2 parts have room for (a model's
    // planes are 16 bytes a spaxel, its parts 12 bytes a tile of at least 16
    // spaxels: in practice all of them)
    TileScratch sc;
    size_t per = (size_t)0x7fffffff / ts.tiles, room = L.pl_bytes;
    char *scratch = (char *)ws + L.pl_off;
    // A small batch in the shape that chi2 is bound to leaves SMs idle: where
    // the batch's own shape (its size rounded up to a power of two: fits call
    // with all sizes, and the shapes are remembered) is estimated at 1 / 1.7 of
    // the cost, the residuals come in that shape and are summed afterwards (a
    // launch of 6 - 9 us).
    TileShape own;
    const size_t np = (size_t)g.nx * g.ny, rbytes = resid ? 0 : al256(2 * np * sizeof(float) * (size_t)n);
    bool two = false;
    if (chi2 && (size_t)n * ts.tiles < 304 &&
        rbytes + (size_t)n * (ts.tiles * sizeof(double) + sizeof(unsigned)) <= room) {
        int m = 1;
        while (m < n) m *= 2;
        two = tile_shape(g, m, false, &own) && tile_cost(g, ts, m) > 1.7 * own.cost;
    }
    float *sums = resid;
    if (two && !resid) {
        sums = (float *)scratch;
        scratch += rbytes;
        room -= rbytes;
    }
    if (timer && (e = timer->mark(st)) != cudaSuccess) return cuda_fail(e, "split evaluator: timing event");
    if (chi2 && ts.tiles > 1) {
        per = std::min(per, room / ((size_t)ts.tiles * sizeof(double) + sizeof(unsigned)));
        per = std::min(per, (size_t)n);
        sc.part = (double *)scratch;
        sc.arrived = (unsigned *)(scratch + per * ts.tiles * sizeof(double));
        e = cudaMemsetAsync(sc.arrived, 0, per * sizeof(unsigned), st);
        if (e != cudaSuccess) return cuda_fail(e, "split evaluator: clearing the arrival counters");
    }
    if (timer && (e = timer->mark(st)) != cudaSuccess) return cuda_fail(e, "split evaluator: timing event");
    if (two) {
        gbk_status s = launch_tile(g, own, n, params, obs, maps, nullptr, sums, TileScratch(), batch, 0, st);
        if (s || (s = launch_tile_resid_sum(g, ts, n, params, sums, chi2, sc, batch, 0, st))) return s;
        if (timer) timer->launches += 2;
    }
    for (size_t m0 = 0; m0 < (size_t)n && !two; m0 += per) {
        const gbk_status s =
            launch_tile(g, ts, (int)std::min(per, (size_t)n - m0), params + m0 * GBK_NPAR, obs,
                        maps ? maps + 3 * np * m0 : nullptr, chi2 ? chi2 + m0 : nullptr,
                        resid ? resid + 2 * np * m0 : nullptr, sc, batch, (int)m0, st);
        if (s) return s;
        if (timer) ++timer->launches;
    }
    if (timer && (e = timer->mark(st)) != cudaSuccess) return cuda_fail(e, "split evaluator: timing event");
    return GBK_OK;
}

}  // namespace gbk

using namespace gbk;

extern "C" gbk_status gbk_split_stage_times(const gbk_geom *gin, int32_t n_models, const double *params,
                                            const gbk_obs *obs, double *chi2, void *workspace, size_t ws_bytes,
                                            float *stage_ms, int32_t *launches, void *stream)
{
    Geom g;
    gbk_status s = derive_geom(gin, &g);
    if (s) return s;
    if (n_models < 1) return fail(GBK_EINVAL, "n_models must be >= 1");
    if (!stage_ms) return fail(GBK_EINVAL, "stage_ms is NULL");
    if ((s = check_device_ptr(params, "params", 8)) || (s = check_device_ptr(chi2, "chi2", 8)) || (s = check_obs(obs)))
        return s;
    if (workspace && (s = check_device_ptr(workspace, "workspace", 256))) return s;
    cudaStream_t st = (cudaStream_t)stream;
    SplitTimer timer;
    s = launch_split(g, n_models, params, obs, nullptr, chi2, nullptr, workspace, ws_bytes, st, &timer);
    cudaError_t e = cudaSuccess;
    if (!s && timer.n > 0) e = cudaEventSynchronize(timer.ev[timer.n - 1]);
    if (!s && e == cudaSuccess && (e = cudaEventElapsedTime(&stage_ms[0], timer.ev[0], timer.ev[1])) == cudaSuccess &&
        (e = cudaEventElapsedTime(&stage_ms[1], timer.ev[1], timer.ev[2])) == cudaSuccess) {
        stage_ms[2] = 0.f;
        if (launches) *launches = timer.launches;
    }
    timer.release();
    if (s) return s;
    if (e != cudaSuccess) return cuda_fail(e, "split stage times");
    return ok();
}
