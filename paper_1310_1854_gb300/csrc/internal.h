// Internal declarations shared by the host builder, the C-ABI layer and the
// CUDA kernels of libvgrid. Not part of the public interface (include/vgrid.h).
#pragma once

#include <vector_types.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <functional>
#include <vector>

namespace vg {

// Host results of the cell construction, in the library's internal cell order.
struct CellsOut {
    std::vector<int64_t> off;   // CSR offsets, M + 1
    std::vector<int32_t> idx;   // neighbour ids (internal) and walls -1..-6
    std::vector<double> vol;    // cell volumes
    std::vector<double> bbox;   // 6 per cell
    // device copies of off, idx and bbox where the GPU construction leaves
    // them, for the caller to free; else NULL
    int64_t *d_off = nullptr;
    int32_t *d_idx = nullptr;
    double *d_bbox = nullptr;
};

struct BlocksOut {
    int32_t dim[3] = {1, 1, 1};
    std::vector<int64_t> off;   // K + 1
    std::vector<int32_t> idx;   // internal cell ids
};

int build_cells(const double *sites, int64_t M, const double *box, int threads, CellsOut &out, std::string &err);
int build_cells_into(const double *sites, int64_t M, const double *box, int threads, const std::vector<int32_t> *ids,
                     std::vector<std::vector<int32_t>> &nbr, double *volume, double *bbox, std::string &err);
void cells_to_csr(const std::vector<std::vector<int32_t>> &nbr, CellsOut &out);
// GPU construction (build_gpu.cu); cells the device could not hold are rebuilt
// on the host. Returns 0, or -1 with err set.
int build_cells_gpu(const double *sites, int64_t M, const double *box, int threads, CellsOut &out, std::string &err,
                    int64_t *host_fallback_cells);
// cells sorted by the Morton code of their site (21 bits per axis); the
// sorted codes go to *codes if given
void morton_order(const double *sites, int64_t M, const double *box, std::vector<int32_t> &perm,
                  std::vector<uint64_t> *codes = nullptr, int threads = 0);
// fn(begin, end) over [0, n) split into contiguous ranges on up to `threads`
// host threads (0: all cores); ranges of fewer than `grain` items stay on
// one thread
void parallel_for(int64_t n, int threads, int64_t grain, const std::function<void(int64_t, int64_t)> &fn);
// blocks per axis of the block lists
void block_dims(const double *box, int64_t M, double blocks_per_site, int32_t *dim);
void build_blocks(const double *box, const std::vector<double> &bbox, int64_t M, double blocks_per_site,
                  BlocksOut &out, int threads = 0);
// GridDev::ushift of a box whose `scale` is given: 0 where the products of two
// lengths in it are ordinary float32 numbers, else unit is about 1 / scale
inline int unit_shift(double scale) {
    const int e = std::ilogb(scale);
    return e >= -20 && e <= 40 ? 0 : -std::min(std::max(e, -120), 120);
}

}  // namespace vg

// ---------------------------------------------------------------------------
// Device-side view of one grid. Plain data, passed by value to kernels or
// stored in an array for batched launches. Cells are in the library's
// internal (Morton) order.
//
// cells    absolute cell blocks (float64 searches of a whole cell), float4: cell i
//          starts at A_i with a header (bits of the caller's id, bits of the
//          neighbour count c, rho, bits of F_i) followed by c records (x, y, z
//          of the neighbour's site, bits of the neighbour's offset A_j, or of
//          a wall id -1..-6).
// rel      relative cell blocks (float32 search), float4: cell i starts at F_i
//          (even) with (x, y, z of p_i, bits of the record count c4) and
//          (bits of the caller's id, rho, N1max, bits of A_i), followed by c4
//          records: (fl(p_j - p_i) as float32, bits of F_j) for every cell
//          neighbour j, nearest first, then NaN records up to c4 = max(4, an even count).
//          N1max bounds |fl(p_j - p_i)|_1 over the records from above.
// site[i]  float4 (x, y, z, bits of F_i): positions for C(r) and ray starts.
// perm[i]  caller's id of internal cell i.
// blk_off, blk_rec  block lists of Sect. 2.3: for every block, records
//          (x, y, z of a site, bits of its internal id) of the cells whose
//          bounding box overlaps the block.
// ---------------------------------------------------------------------------
struct GridDev {
    const float4 *site;
    const float4 *cells;
    const float4 *rel;
    const int32_t *perm;
    const int32_t *blk_off;
    const float4 *blk_rec;
    double lo[3], hi[3];      // domain box
    double bscale[3];         // blocks per unit length along each axis
    int64_t lokey[3], hikey[3];        // order keys of lo and hi (exact box test)
    float flo_hi[3], flo_lo[3];        // lo as float pairs
    float fbscale[3];                  // bscale in float32
    float fbw[3];                      // block width in float32; block (i, j, k) has the
                                       // centre flo_hi + (i + 1/2) fbw (float32 operations),
                                       // and its list is ordered by distance from it
    const float *dens;                 // coarse grid of (sites per unit volume)^(1/3), for the ray order
    int32_t ddim[3];                   // its cells per axis
    float dscale[3];                   // its cells per unit length
    int32_t ospatial;                  // ray order: start-cell ranges per length bin (1: length only)
    int32_t bdim[3];
    int32_t M;
    float kappa;
    int32_t zmax;             // zero-length steps in a row before the epsilon nudge
    double eps64;             // epsilon nudge, float64 path
    double eps32;             // epsilon nudge, float32 path
    double scale;             // max |coordinate| of the box + diagonal
    int64_t max_steps;
    int32_t domain;           // VGRID_DOMAIN_BOX or VGRID_DOMAIN_SPHERE
    float lslack;             // C(r): off the bound that stops the scan of a block list. 2^-70 covers square
                              // roots of sums rounded in the subnormal range; infinite (no stop) where a
                              // sum of squares may overflow, whose root would bound nothing
    float unit;               // power of two that the float64 form's float32 search takes lengths by
    int32_t ushift;           // unit = 2^ushift
    double sph[4];            // spherical domain: centre and radius
};

// Per-ray record written by the start-cell kernel (full warps, where the
// float64 set-up is cheap) and read once by the traversal kernel when the
// ray starts (64 bytes).
struct RayPrep {
    int32_t cell;             // offset of the start cell's relative block; -1 outside the box,
                              // -2 direction not unit
    int32_t wall;             // wall the ray leaves through (Eq. 5), -1..-6
    float tmax_hi, tmax_lo;   // distance to that wall, as a float pair
    float r0_hi[3], r0_lo[3]; // origin as float pairs
    float k_hi[3], k_lo[3];   // direction as float pairs
};

// The same for the float64 form.
struct RayPrep64 {
    int32_t cell;             // as in RayPrep: offset of the start cell's relative block, or -1, -2
    int32_t wall;             // the wall ahead, -1..-6 or -7 (sphere), where t_lo and t_hi name one
    float t_lo, t_hi;         // bounds on the distance to the domain's boundary from the origin as the
                              // float64 form evaluates it anywhere on the path; t_hi is infinite where
                              // two walls are too close to call
    double o[3], d[3];        // origin and direction
};
static_assert(sizeof(RayPrep) == 64 && sizeof(RayPrep64) == 64, "start records");

// A batch work descriptor: rays of one grid.
struct RaySetDev {
    const double *origin;
    const double *dir;
    void *tau;                // float (float32 form) or double (float64 form), nullable
    int32_t *status;          // nullable
    RayPrep *start;           // per-ray start records - work buffer
    int64_t n;
    int64_t first;            // global index of the first ray of this set
    int32_t grid;             // index into the GridDev array
    int32_t pad;
};

// Counters accumulated on the device; mirrors vgrid_stats.
struct StatsDev {
    unsigned long long rays, crossings, decisions, rechecks, fallbacks, zero_steps, step_limit, outside, bad_dir;
    unsigned long long cursor;  // segment mode: chunks handed out, read back with the counters
};


// What the allocation-free entry point (noalloc.cu) needs from a grid.
struct vgrid;
namespace vg {
struct GridView {
    int device;
    int sms;
    const GridDev *d_desc;
    GridDev hd;  // host copy of *d_desc
};
int grid_view(const struct vgrid *g, GridView *out);  // 0, or -1 for a host-only grid
void set_error(const std::string &msg);              // message for vgrid_last_error()
}  // namespace vg
