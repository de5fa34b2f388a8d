// Host-side table and raster builders.
#pragma once

#include <vector>

#include "vpmc_internal.cuh"

namespace vpmc {

// curve15 = {hu[5], density[5], spr[5]}
void build_tables(const double* curve15, TablesImage* img);
double pmma_stopping_power_ratio(double kinetic_mev);
// Raster of an opening's polygon, kRaster x kRaster cells.  Points outside it
// are at least `margin` from the boundary.
struct Raster {
    std::vector<unsigned char> cells;      // 0 outside, 1 inside, 2 near an edge
    std::vector<float> lower;              // lower bound of the distance to the boundary
    std::vector<uint16_t> near;            // edge nearest to the cell's centre
    std::vector<uint32_t> local;           // cells near an edge: the crossing-number test's edges (0: all)
    float lo[2], inv[2];                   // origin, 1 / cell size
    float diag;                            // cell diagonal (plus a margin)
};
void build_raster(const double* xy, int n, double margin, Raster* out);
// Signed curvature (1/mm) of each polygon vertex: the turning angle at the
// vertex over half the sum of its two edges, positive where the region inside
// the polygon is locally convex (either vertex order).
void polygon_curvature(const double* xy, int n, float* kappa);
void hu_curve_props(const double* curve15, double hu, double* rho, double* spr);

}  // namespace vpmc
