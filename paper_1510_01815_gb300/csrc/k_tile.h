// k_tile.h -- launcher of the one-kernel evaluator (k_tile.cu).
#pragma once

#include "gbk_internal.cuh"
#include "k_split.h"

namespace gbk {

constexpr int kTileMaxR = kSplitMaxR;  // largest PSF radius the kernel is compiled for

// A model's image cut into tiles of tx x ty data spaxels, one CTA each.
struct TileShape {
    int tx, ty;            // data spaxels per tile, multiples of 4
    int tiles_x, tiles;    // tiles per row, tiles per model
    int threads;           // CTA size
    size_t smem;           // dynamic shared memory per CTA
    double cost;           // estimated cost of the call (to compare shapes)
};

// chi2 is summed by tiles and threads, so its rounding depends on the shape:
// every call that returns chi2 takes the shape of a batch of this many models,
// whatever its own count, or sums up in that order.  (A fit compares a model's
// chi2 from batches of different sizes; with equal parameters they must be
// equal to the bit.)
constexpr int kTileChi2Batch = 2048;

// The cheapest shape for n_models models (`whole`: one tile per model, two
// CTAs or more per SM); false where the kernel does not serve the geometry or
// no such shape fits.
bool tile_shape(const Geom &g, int n_models, bool whole, TileShape *out);

// A shape's estimated cost for n_models models.
double tile_cost(const Geom &g, const TileShape &s, int n_models);

// chi2 parts of `tiles` tiles per model: doubles, then arrival counters
// (zero at the start and left zero).  Not needed for one tile per model.
struct TileScratch {
    double *part = nullptr;
    unsigned *arrived = nullptr;
};

// Maps, chi2 and residuals (each may be null) of n models; asynchronous.
gbk_status launch_tile(const Geom &g, const TileShape &ts, int n, const double *params, const gbk_obs *obs,
                       float *maps, double *chi2, float *resid, const TileScratch &scratch, const SplitBatch *batch,
                       int m0, cudaStream_t st);

// chi2 of n models from their residuals [n][2][ny][nx], with the bits that
// launch_tile gives in shape ts.
gbk_status launch_tile_resid_sum(const Geom &g, const TileShape &ts, int n, const double *params, const float *resid,
                                 double *chi2, const TileScratch &scratch, const SplitBatch *batch, int m0,
                                 cudaStream_t st);

// A ragged batch's galaxies, every image whole in one CTA.
// Models gal * mpg + s (s < mpg) of the galaxies order[0 .. items / mpg);
// galaxy gal's maps and residuals start at pixel pix_off[gal] * mpg.
struct TileRagged {
    const Geom *geoms;       // device
    const int64_t *pix_off;  // device
    const int32_t *order;    // device
    const double *params;
    const gbk_obs *obs_list; // device, per galaxy (with chi2 or resid)
    const int32_t *skip;     // device, per galaxy: non-zero = left alone (or null)
    float *maps;
    double *chi2;
    float *resid;
    int *work;               // device counter, zero at the start
    int items, mpg;
};
// The CTA size that serves the galaxy and its shared memory; 0: not served.
int tile_ragged_threads(const Geom &g, size_t *smem);
// `overlap`: the launch before it in the stream is another of the same call,
// of this kernel or a persistent one of the cluster evaluator.
gbk_status launch_tile_ragged(const TileRagged &a, int threads, size_t smem, bool overlap, cudaStream_t st);

}  // namespace gbk
