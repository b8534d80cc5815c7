// Launch plans of the TMA step kernel (mmod_step_tma.cu).
#pragma once
#include <cuda.h>

#include "mmod.h"

namespace mmod {

constexpr int kMaxTmaVariants = 12;
// The 64 x 16 staged variant: what the batch, persistent and work-claiming
// forms are compiled for, and what a handle runs when no other tile shape
// serves its grid better (TmaShape).
constexpr int kTmaDefaultVariant = 2;

// Tile shapes of the compiled variants: TX x TY points, halo rows of `pitch`
// floats.  Injection tables are bucketed per tile, so a handle keeps tensor
// maps and tables per shape it runs (ensure_shape).
struct TmaShape {
    int tx, ty, pitch;
};
constexpr int kNumShapes = 4;
constexpr TmaShape kTmaShapes[kNumShapes] = {{64, 16, 72}, {48, 20, 56}, {40, 24, 52}, {32, 32, 40}};

// Source points the imaging form takes: one per thread of its smallest block.
constexpr int kMaxImageSources = 240;

struct TmaPlan {
    int variant = 0;                // index into the compiled variants
    int shape = 0;                  // index into kTmaShapes
    bool has_g = false;             // compiled with the g^n output (StepArgs::gout)
    bool has_image = false;         // compiled with the imaging form (StepArgs::image)
    int tiles_x = 0, tiles_y = 0;   // x-y tiles covering the plane
    int zchunks = 0;                // z-ranges per tile column
    int zlen = 0;                   // planes per z-range (last one may be shorter)
    int grid = 0;                   // CTAs launched
    int block = 0;                  // threads per CTA
    int smem = 0;                   // dynamic shared memory per CTA, bytes
    int occupancy = 0;              // resident CTAs per SM
    int slots = 0;                  // resident CTAs on the device (SMs x occupancy)
    int claim = 0;                  // > 0: work-claiming launch with units of this many planes
};

struct Geom;
// Units and grid of a work-claiming launch of plan (false: the plan's variant
// has no work-claiming form or claim is off).
bool claim_geom(const TmaPlan &plan, int nz, Geom *g, int *units, int *grid);

int tma_variant_count();
const char *tma_variant_name(int v);

// Tensor maps of one padded volume buffer for a tile shape: the halo box
// (u^n) and the tile box (u^{n-1}, c, and the planes of u^n without halo).
struct VolMaps {
    CUtensorMap halo, own;
};
bool encode_maps(const mmod_config &cfg, int nxp, const float *buf, int shape, VolMaps *m);

// Fills one plan per compiled variant.  False when the TMA kernels cannot
// run (the caller then uses the plain kernel).
bool make_tma_plan(const mmod_config &cfg, TmaPlan plans[]);
// The variant a handle runs by default: the tile shape and z split of least
// cost for its grid (rule beside the definition).
int auto_tma_variant(const TmaPlan plans[]);
bool tma_variant_has_batch(int v);

}  // namespace mmod
