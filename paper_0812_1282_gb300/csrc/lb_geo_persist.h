// Host entry points of the obstacle steps' tile lists and multi-step forms
// (lb_geo.cu).
#pragma once

#include <vector>

#include "lb_internal.h"

namespace lbfe {

// Tiles of the per-step form, 32 columns x `rows`: those with a fluid or wall
// node, the ones whose fluid touches a solid node first and marked by their
// sign bit (they take longer).  FP32 takes 8 rows while all tiles are
// resident at once (three to an SM), else 4, of which more fit (us per step with 8
// and 4 rows of channels with so many tiles of 8 rows: 230 (1000 x 120) 3.7 and
// 5.2, 428 5.0 and 5.4, 482 7.3 and 5.6, 735 8.7 and 8.2, 1011 (2000 x 200) 12.2
// and 9.8).  FP64 takes 4: the FP64 pipe of each SM is the bound and smaller tiles
// share the work out more evenly (401 x 77, before the extra warps: 10.2 with 4,
// 13.9 with 8, 12.6 with 2).  geo_tile_capacity: the most entries a list can have.
constexpr int kGeoTileIndex = 0x7fffffff;
struct GeoTiles {
    int rows;
    std::vector<int> list;
};
GeoTiles make_geo_tiles(int precision, int sm_count, const unsigned char* cls, int nx, int ny,
                        int walls);
size_t geo_tile_capacity(int nx, int ny);

// Persistent multi-step obstacle step (a cooperative launch of one CTA per
// tile for n_steps steps, step s reading buffer parity0 ^ (s & flip));
// flags: geo_tiles(nx, ny) ints, done: one int, all zero between launches.
// geo_persist_occupancy: resident CTAs per SM (0 on error).
int geo_tiles(int nx, int ny);
int geo_persist_occupancy(int precision, int coll);
int launch_geo_persist(int precision, int coll, const DomDesc& d, int parity0, int flip,
                       int n_steps, int* flags, int* done, void* stream);
// Two steps of an obstacle domain in one launch (temporal blocking): reads
// buffer `parity`, writes the other (which then holds the state two steps
// on).  prepare_geo_step2 opts the kernel in to its shared memory (once per
// device, outside any stream capture).
int launch_geo_step2(int precision, int coll, const DomDesc& d, int parity, void* stream);
int prepare_geo_step2();

}  // namespace lbfe
