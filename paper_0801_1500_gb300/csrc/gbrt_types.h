// Internal device-side views of scenes, grids and frames, shared by the host
// orchestration code and the kernels of libgbrt (never exposed in the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gbrt.h"

namespace gbrt {

// Error bits of the context's device error word.
enum : uint32_t {
    ERR_DDA_STEPS = 1u,      // a grid walk exceeded nx + ny + nz + 3 steps
    ERR_SCENE_DATA = 2u,     // non-finite / non-positive scene values (device upload path)
    ERR_QUEUE_TIMEOUT = 4u,  // reserved: a bounded wait ran out (no kernel of this version waits)
    ERR_GRID_CAPACITY = 8u,  // a device-side grid rebuild outgrew its item buffer
};

// Scene in the device layout: one record per object, indexed by global id
// (spheres 0..S-1, then cylinders S..S+C-1), the same shape for both kinds so
// a single branch-free test serves both (a sphere is a cylinder record with a
// zero axis and zero length):
//   obj    float4 [2 (S+C)]  (p0 xyz, radius), (unit axis xyz, length)
//   obj64  double2[4 (S+C)]  (p0x, p0y), (p0z, radius), (ax, ay), (az, length)
//   bs     float4 [S+C]      ball around each object (centre, radius): a sphere
//                            itself, or the ball around a tube with its radius
//                            negated (16 bytes to reject a candidate from)
//   color  uint32 [S+C] palette index; palette float [K*3]
struct SceneDev {
    int32_t S, C, K, pad;
    const float4* obj;
    const double2* obj64;
    const float4* bs;
    const uint32_t* color;
    const float* palette;
};

// Uniform grid. balls are the scene's objects sorted by the cell of a grid with
// half as many cells an axis (bn = ceil(n / 2), same corner, h doubled) that
// holds their centre, x fastest: those of cells (x0..x1, y, z) are
// [bstart[(z bny + y) bnx + x0], bstart[(z bny + y) bnx + x1 + 1]). A tube's
// ball holds only the part outside its spheres (radius negated; 0: no such
// part). They are copies: a scene that was updated since, or another one of as
// many objects, is rendered without them (FrameDev::stale). rho is the reach of the AO rays' near pass (0: not used), rmax the
// largest distance of an object's point from the centre it was sorted by.
// cells[c] = (first item, item count) of cell
// c = (z * ny + y) * nx + x; items are global object ids, in the order the
// scatter pass left them (no result depends on the order).
struct GridDev {
    float lo[3], hi[3], h[3], inv_h[3];
    double lo64[3];
    // bounding sphere of all objects (centre xyz, radius): walks are clipped to
    // it, so rays skip the empty corners of the grid box
    float bs[4];
    double bs64[4];
    int32_t n[3];
    int32_t empty;
    int64_t ncells;
    int64_t nitems;  // length of the item buffer
    const uint2* cells;
    const uint32_t* items;
    const float4* balls;
    const uint32_t* bstart;
    const float4* cut;  // the same balls by object id
    int32_t bn[3];
    int32_t nballs;
    float rho, rmax;
    float density;  // objects per volume of the grid box
};

// Everything one frame needs, in the precision each path reads.
struct FrameDev {
    SceneDev scene;
    GridDev grid;
    // camera (double) -- the float path rounds the primary ray from these
    double eye[3], dir[3], up[3], right[3];
    double half_w, half_h;
    double inv_w, inv_h;  // 1/W, 1/H
    double dir_unit[3];   // dir / |dir|
    float dir_f[3], up_f[3], right_f[3];
    float half_w_f, half_h_f, inv_w_f, inv_h_f;
    // the float path's primary rays as float-float pairs (value = hi + lo,
    // |lo| <= half an ulp of hi). The part that varies with pixel (i, j) is
    // affine in it, a0 + i ai + j aj: the orthographic origin (direction
    // dir_unit), or the pinhole direction before normalisation (origin eye)
    float a0_hi[3], a0_lo[3], ai_hi[3], ai_lo[3], aj_hi[3], aj_lo[3];
    float dir_hi[3], dir_lo[3], eye_hi[3], eye_lo[3];
    int32_t cam_kind;
    int32_t W, H, spp;
    int32_t shadows;       // 1: one shadow ray per light the surface faces
    int32_t jobs_per_hit;  // AO samples + shadow rays of one hit
    uint32_t jph_magic;    // ceil(2^32 / jobs_per_hit) when jobs_per_hit > 1 (division by multiply)
    uint32_t frame;
    uint32_t seed_lo, seed_hi;
    int32_t precision;
    // shading
    int32_t nl;
    int32_t phong_n;  // the Phong exponent where it is a whole number from 1 to 1024, else 0
    double ldir[GBRT_MAX_LIGHTS][3];
    double lI[GBRT_MAX_LIGHTS];  // intensity * scale
    float ldir_f[GBRT_MAX_LIGHTS][3];
    float lI_f[GBRT_MAX_LIGHTS];
    double sky_kao, k_d, k_s, phong;
    float sky_kao_f, k_d_f, k_s_f, phong_f;
    double eps, ao_maxdist;
    float eps_f;
    float ao_maxdist_f;
    double bg[3];
    float bg_f[3];
    // outputs (device). Pixel q of the rendered raster writes its colour at
    // out_rgb + 3 (q - rgb_q0). With supersampling (aa = m > 1) the rendered
    // raster is the m-times finer one (W, H, row0, rows count its pixels),
    // out_rgb is the library's buffer for the band's finer rows, and the
    // resolve pass box-filters it into out_final ((W/m) x (H/m) pixels).
    void* out_rgb;
    uint32_t* out_ids;
    uint32_t* out_vis;
    void* out_final;
    int64_t rgb_q0;
    int32_t aa;
    // grid rebuilt on the device: its current geometry, copied over `grid`
    // before the frame's kernels run (null for grids built on the host)
    const GridDev* grid_src;
    // rows [row0, row0 + rows) of the image are rendered (a band, or all rows);
    // their tiling into primary-ray work items (tile_w x tile_h = 32)
    int32_t row0, rows;
    int32_t tiles_x, tiles_y;
    int64_t hit_base;  // first slot of this frame's region of the hit buffers
    int32_t stale;     // 1: the grid's balls are of another geometry than the scene's
    // near pass: 1 when it looks for this frame's near occluders; the frame's
    // words in the job masks (mask_words a hit, 16 jobs a word)
    int32_t near_pass;
    int32_t mask_words;
    int32_t rec_words;  // words of one tile record
    int64_t mask_base;
};

// Up to rec_words words of 16 jobs of the hits of one primary work item (tile),
// as the near pass and the AO walk see them: the hits' first slot and number,
// their frame, the first job word, and how far the near pass looked.
struct TileRec {
    int64_t slot;
    int32_t n;
    int32_t frame;
    int32_t word;
    float rho;
};

// One batch of frames as the render kernels see it (a kernel parameter).
//   frames    [n] descriptors (device)
//   tile_off  [n + 1] prefix sums of primary work items (device)
//   hit_count [n] hits appended by the primary pass, per frame
//   job_off   [n + 1] prefix sums of AO rays (hits x samples) per frame
//   hit_off   [n + 1] prefix sums of hits per frame
//   hits      2 records per hit (FP32: float4 pairs; FP64: 4 double2), at
//             frames[f].hit_base + h:  (origin xyz, pixel)  (normal xyz, object id)
//   hits32    what the AO walk reads, float4 pairs in both precisions: `hits`
//             itself in FP32; in FP64 the same layout with the origin relative
//             to the grid's lower corner
//   vis       escaped AO samples per hit slot
//   lmask     per hit slot, bit l set when the shadow ray toward light l escaped
//   queue     [0] next primary work item, [1] next AO ray (or unit), [2] next
//             tile of the near pass, [3] finished CTAs of the primary pass, then
//             the number of rays an AO warp claims at once
// With a near pass (tiles not null):
//   tiles     records of the work items with hits
//   ntiles    their number
//   masks     per hit and 16 jobs: low half the jobs whose ray still has to
//             walk, high half those of them that walk from the start
//   units     (record << 8 | group of 4 of the frame's jobs) with a ray left to walk
//   nunits    their number
struct BatchDev {
    const FrameDev* frames;
    const long long* tile_off;
    unsigned int* hit_count;
    unsigned long long* job_off;
    unsigned long long* hit_off;
    void* hits;
    void* hits32;
    unsigned int* vis;
    unsigned int* lmask;
    unsigned long long* queue;
    unsigned int* err;
    TileRec* tiles;
    unsigned int* masks;
    unsigned long long* units;
    unsigned long long* nunits;
    unsigned long long* ntiles;
    int64_t hit_cap;  // hit slots (records, vis, lmask) of the batch
    int64_t tile_cap, mask_cap, unit_cap;  // lengths of tiles, masks and units
    int32_t nframes;
    int32_t tile_w, tile_h;
    int32_t refill;
    int32_t ao_warps;  // warps of the AO walk
    int32_t parts;     // lanes that share a primary ray (1, 2, 4 or 8)
};

}  // namespace gbrt
