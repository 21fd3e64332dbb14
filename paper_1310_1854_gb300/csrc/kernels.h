// Kernel tables and host-callable launch helpers of libvgrid (internal).
#pragma once

#include <cuda_runtime.h>

#include "internal.h"

namespace vg {

enum { MODE_TAU = 0, MODE_SEGS = 1, MODE_GRAD = 2, MODE_INTERACT = 3, NUM_MODES = 4 };

// Segment lists in one traversal. A ray's segments go, in path order, into
// chunks of kSegChunk slots of a work buffer; each chunk records its ray and
// its position in that ray's list, so once the counts have been scanned a
// compaction kernel can copy every chunk to its place in the CSR arrays
// independently of the others. Chunks are handed to the lanes of a warp from
// a page of kSegPage chunks that the warp takes from one global cursor, so
// the cursor sees one atomic per kSegPage chunks. A slot is int2 (cell,
// float32 length) or int4 (cell, 0, float64 length as low and high words).
constexpr int kSegChunk = 8;
constexpr int kSegPage = 32;  // >= 32: one ballot's requests always fit in what is left plus one page

struct TraceArgs {
    const GridDev *grids;     // one descriptor per grid
    const RaySetDev *sets;    // one per (grid, rays) set
    int32_t nsets;
    int64_t total;            // rays over all sets
    unsigned long long *queue;
    StatsDev *stats;
    // segment mode
    int64_t *seg_off;         // segment count per ray (scanned afterwards)
    void *seg_slots;          // chunk slots (kSegChunk per chunk)
    int2 *chunk_meta;         // per chunk: (ray, position in the ray's list); ray -1: unused
    unsigned long long *chunk_cursor;  // chunks handed out (zeroed by the caller)
    int64_t chunk_cap;        // chunks in the buffer; segments beyond are counted, not stored
    const float *dL_dtau;
    float *dL_drho;
    // interaction mode
    const float *tau_int;     // optical depth at which each ray interacts
    const float *weight;      // package weight per ray (nullable: 1)
    int32_t *int_cell;        // caller id of the interaction cell, -1 if the ray escapes
    float *int_s;             // distance from the origin to the interaction point (or the exit)
    float *absorbed;          // per cell (caller ids), accumulated; nullable
    // single-grid launches read the grid and the ray set from here (kernel
    // parameter space) instead of from `grids` / `sets`
    GridDev g1;
    RaySetDev s1;
    const int32_t *order;     // nullable: queue position -> ray (longest predicted first)
};


// Shared memory of a traversal block, per warp: the queue of rays to start
// (records, ray indices, head and count, per-ray scalars: the adjoint's
// dL/dtau, interaction's tau_int and weight, a batch's ray set) and the float32
// form's per-ray values.
constexpr int kFetch = 32;    // rays a warp's queue holds
constexpr int kRayVals = 11;  // per-ray floats of the float32 form
constexpr int trace_queue_bytes(int mode, bool batch) {
    return kFetch * ((int)sizeof(RayPrep) + 8 + 4 * (mode == MODE_GRAD ? 1 : mode == MODE_INTERACT ? 2 : 0) +
                     (batch ? 4 : 0)) + 16;
}
constexpr int trace_warp_bytes(bool fp64, int mode, bool batch) {
    return trace_queue_bytes(mode, batch) + (fp64 ? 0 : 32 * 4 * kRayVals);
}

// a traversal kernel and the shared memory that a block of it takes per warp
struct TraceFn {
    const void *fn;
    int warp_bytes;
    size_t smem(int block) const { return (size_t)(block / 32) * warp_bytes; }
};

// fn[fp64][mode]: single-grid trace kernels of one lanes-per-ray value
// (nullptr if absent); batch: the float32 tau kernel over many grids
struct KernelSet {
    // fn[0]: float32 form, fn[1]: float64 form, fn[2]: float32 form with
    // exact lengths
    const void *fn[3][NUM_MODES];
    const void *batch;
    TraceFn get(int row, int mode) const { return {fn[row][mode], trace_warp_bytes(row == 1, mode, false)}; }
    TraceFn get_batch() const { return {batch, trace_warp_bytes(false, MODE_TAU, true)}; }
};

// the tau kernel and launch shape of a call of N rays on g (api.cu), with g's
// device current
TraceFn pick_trace(const struct ::vgrid *g, int row, int64_t N, int *block, int *blocks);

void kernel_table_lpr1(KernelSet &k);
void kernel_table_lpr2(KernelSet &k);
void kernel_table_lpr4(KernelSet &k);
void kernel_table_lpr8(KernelSet &k);

// auxiliary kernels (aux.cu)
// kernels launched by this library in this process (every launch helper
// adds the kernels it launched)
void count_launches(int64_t n);
int64_t launches_so_far();

cudaError_t launch_put_grid(GridDev *d, const GridDev &g, cudaStream_t s);
cudaError_t launch_enter(const double *origin, const double *dir, int64_t N, const GridDev *gp, double *out, int sms,
                         cudaStream_t s);
// what the start-cell kernel writes per ray (see locate_kernel)
enum { PREP_CELL32 = 0, PREP_FP32 = 1, PREP_FP64 = 2, PREP_CELL64 = 3 };
// Longest-predicted-first ray order. A persistent launch ends when its last
// ray does, so long rays handed out late leave most lanes idle at the end;
// handing the longest out first fixes that. The start-cell kernel estimates
// each ray's crossings (sum of the coarse (sites per volume)^(1/3) grid at 8
// points of its in-box segment, times the segment length) and counts rays
// per bin; a scan and a scatter turn the bins into the permutation the
// traversal takes its rays from, highest bin first. For a grid whose blocks
// fit in L2 the bin is the quarter-octave of the estimate; for a larger one
// it is (half-octave of the estimate, one of 16 ranges of the start cell's
// Morton index), so that the rays in flight at a time start in one part of
// the grid and share more of L2.
constexpr int kOrderBins = 256;
struct RayOrder {
    uint8_t *bin;     // per ray
    uint32_t *hist;   // kOrderBins counts, then kOrderBins cursors (zeroed by the caller)
    int32_t *order;   // queue position -> ray
};
// One launch of the start-cell kernel. sets: device, nsets of them, or NULL for
// the one set `one`. bin, hist: with them the ray order's bins and their counts
// come too (PREP_FP32 and PREP_FP64). queue, stats: cleared for the traversal
// that follows on the stream (nullable: host-pipelined chunks keep adding up
// their counters).
struct LocateArgs {
    const GridDev *grids;
    const RaySetDev *sets;
    int32_t nsets;
    RaySetDev one;
    int64_t total;
    int32_t *out_caller;
    uint8_t *bin;
    uint32_t *hist;
    unsigned long long *queue;
    StatsDev *stats;
};
cudaError_t launch_locate(const LocateArgs &a, int prep, int sms, cudaStream_t s);
// bins -> permutation (scan of the counts, longest bin first, and scatter)
cudaError_t launch_order(const RayOrder &ord, int64_t total, int sms, cudaStream_t s);
cudaError_t launch_permute_density(const float *rho_caller, const int32_t *perm, const float4 *site, int64_t M,
                                   float4 *cells, float4 *rel, cudaStream_t s);
// Device arrays of a grid from its cells (layout.cu), on the current device.
// site4, perm, off, idx, bbox: host, in the internal cell order; d_off, d_idx,
// d_bbox: the same on the device where the cell construction left them
// there, else NULL.
struct LayoutIn {
    int64_t M;
    int sms;
    const double *box;
    float unit;                 // GridDev::unit
    int32_t bdim[3], ddim[3];   // block grid, coarse density grid
    const float4 *site4;        // (x, y, z, -) per cell
    const int32_t *perm;
    const int64_t *off;
    const int32_t *idx;
    const double *bbox;
    const int64_t *d_off;
    const int32_t *d_idx;
    const double *d_bbox;
};
struct LayoutOut {
    float4 *site, *cells, *rel, *blk_rec;
    int32_t *perm, *blk_off;
    float *dens;
    int64_t ncells, nrel, blk_records;  // float4 records of cells, rel, blk_rec
    int64_t entries;                    // entries of all block lists, without padding
    double seconds[3];                  // copies in, block lists, cell blocks
};
enum { LAYOUT_OK = 0, LAYOUT_NOMEM = 1, LAYOUT_CUDA = 2 };
int build_layout(const LayoutIn &in, LayoutOut &out, std::string &err);
// Segment lists in ray order. counts_to_off holds the segments per ray 0..N-1
// and becomes their offsets off[0..N]; then the segments of the chunks the
// traversal took (read from the chunk cursor on the device, at most
// chunk_cap; see kSegChunk) are copied into the CSR arrays, unless off[N]
// exceeds cap (then nothing is written) or chunk_cap is 0 or cell or len NULL.
// coff holds N+1 and inv chunk_cap values of scratch, scan_tmp
// segment_tmp_elems(N).
int64_t segment_tmp_elems(int64_t n);
cudaError_t launch_segment_lists(int64_t *counts_to_off, int64_t N, int64_t chunk_cap, const unsigned long long *cursor,
                                 const int2 *meta, const void *slots, bool fp64, int64_t cap, int64_t *coff,
                                 int64_t *scan_tmp, int32_t *inv, int32_t *cell, void *len, int sms, cudaStream_t s);
// adjoint from segment lists: out[cell[k]] += g[r] * kappa * len[k] for the
// segments k of every ray r (CSR offsets off[0..N])
cudaError_t launch_segments_grad(const int64_t *off, const int32_t *cell, const float *len, int64_t N, const float *g,
                                 float kappa, float *out, int sms, cudaStream_t s);
// exclusive scan of counts[0..n-1] (int64) into off[0..n]; tmp holds
// scan_tmp_elems(n) int64 values
int64_t scan_tmp_elems(int64_t n);
cudaError_t launch_exclusive_scan(int64_t *counts_to_off, int64_t n, int64_t *tmp, cudaStream_t s);

}  // namespace vg
