// Auxiliary kernels of libvgrid: start-cell location (C(r), Sect. 2.3), which
// also clears a call's counters, density reordering and the prefix sum that
// turns per-ray segment counts into offsets.
#include <algorithm>
#include <atomic>

#include "kernels.h"
#include "trace.cuh"

namespace vg {

static std::atomic<int64_t> g_launches{0};
void count_launches(int64_t n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
int64_t launches_so_far() { return g_launches.load(std::memory_order_relaxed); }

__global__ void put_grid_kernel(GridDev *d, GridDev g) { *d = g; }

cudaError_t launch_put_grid(GridDev *d, const GridDev &g, cudaStream_t s) {
    put_grid_kernel<<<1, 1, 0, s>>>(d, g);
    count_launches(1);
    return cudaGetLastError();
}

// Start records for every ray of every set. PREP_CELL32 / PREP_CELL64: C(r0)
// only, written as the caller's id to out_caller (no start record), with
// float32 (rechecked) or float64 distances;
// PREP_FP32: float32 form (cell, direction check, wall exit of Eq. 5 and the
// float pairs of origin and direction); PREP_FP64: float64 form (cell,
// direction check, bounds on the wall exit, origin and direction). The caller's
// id of the cell goes to out_caller if given.
// One instance per kind of record, with the search inlined: the cells alone
// then fit without spills.
// Held to five blocks of 256 threads per SM (48 registers, a few spilled):
// the kernel waits on its loads, and the extra warps hide more of that wait
// than the spilled bytes cost. The cells alone need 40 registers: six blocks
// (10^7 points of the 10^6-site disk 426 -> 405 us; seven spill, 430).
template <int PREP>
__global__ void __launch_bounds__(256, PREP == PREP_CELL32 || PREP == PREP_CELL64 ? 6 : 5)
    locate_kernel(const __grid_constant__ LocateArgs a) {
    uint8_t *const bin = a.bin;
    int32_t *const out_caller = a.out_caller;
    // the work counter and the counters of the traversal that follows (a kernel
    // of its own did this and stored the ray set before: about 3 us per call)
    if (blockIdx.x == 0) {
        constexpr int kCounters = sizeof(StatsDev) / sizeof(unsigned long long);
        if (a.stats && threadIdx.x < kCounters) reinterpret_cast<unsigned long long *>(a.stats)[threadIdx.x] = 0ull;
        if (a.queue && threadIdx.x == kCounters) *a.queue = 0ull;
    }
    __shared__ uint32_t s_hist[kOrderBins];
    if (bin) {
        for (int b = threadIdx.x; b < kOrderBins; b += blockDim.x) s_hist[b] = 0u;
        __syncthreads();
    }
    for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < a.total;
         w += (int64_t)gridDim.x * blockDim.x) {
        const RaySetDev *rs = a.sets ? a.sets + find_set(a.sets, a.nsets, w) : &a.one;
        const int64_t li = w - rs->first;
        const GridDev *gp = a.grids + rs->grid;
        const double *o = rs->origin + 3 * li;
        const LocPt P = loc_point(__ldg(o), __ldg(o + 1), __ldg(o + 2));
        // float32 distances with the proven float64 fallback give exactly the
        // float64 argmin, so both traversal forms start that way; only
        // vgrid_locate's float64 mode (PREP_CELL64) scans in float64
        int m = locate_point<true>(gp, P, PREP != PREP_CELL64, nullptr);
        if (out_caller) out_caller[w] = m >= 0 ? __ldg(&gp->perm[m]) : -1;
        if (PREP == PREP_CELL32 || PREP == PREP_CELL64) continue;
        RayPrep *out = rs->start + li;
        const double *d = rs->dir + 3 * li;
        const double k[3] = {__ldg(d), __ldg(d + 1), __ldg(d + 2)};
        RayPrep p;
        for (int c = 0; c < 3; c++) {
            p.r0_hi[c] = P.h[c];
            p.r0_lo[c] = P.l[c];
            split_pair(k[c], p.k_hi[c], p.k_lo[c]);
        }
        // |k.k - 1| <= 2.000001e-6, in float32 from the pairs (error below
        // 1e-6) unless that is too close to call, then in float64
        float kkf = 0.0f;
        for (int c = 0; c < 3; c++)
            kkf = __fmaf_rn(p.k_hi[c], p.k_hi[c], __fmaf_rn(2.0f * p.k_hi[c], p.k_lo[c], kkf));
        const float dev = fabsf(__fsub_rn(kkf, 1.0f));
        bool unit;
        if (dev <= 1.000001e-6f) {
            unit = true;
        } else if (dev > 3.000001e-6f || !(dev == dev)) {
            unit = false;
        } else {
            const double kk = __dadd_rn(__dadd_rn(__dmul_rn(k[0], k[0]), __dmul_rn(k[1], k[1])), __dmul_rn(k[2], k[2]));
            unit = fabs(kk - 1.0) <= 2.000001e-6;
        }
        if (!unit) m = -2;
        constexpr bool fp64 = PREP == PREP_FP64;
        // the traversal starts from the cell's relative block
        p.cell = m >= 0 ? __float_as_int(__ldg(&gp->site[m]).w) : m;
        // distance to the wall ahead (Eq. 5 for the walls the ray faces), as
        // a float pair: q1 = n/k rounded, the exact remainder n - q1 k by
        // fma, then q2 = remainder / k (relative error a few 2^-48); in a
        // spherical domain the sphere's exit from the origin in float64,
        // split into a float pair
        float th = 3.0e38f, tl = 0.0f;
        int wid = -1;
        // float64 form: bounds on the exit distance that also hold for what it
        // evaluates later from its moved point, which is off the line by up to
        // steps 2^-53 |coordinates| (it trusts them up to 2^15 steps): a wall's
        // distance then moves by that over |k_c|, the sphere's root, whose
        // square root may have a small argument, by up to 2^-18 of the scale
        const float scale = (float)gp->scale;
        float w_lo = 3.0e38f, w_hi = 3.0e38f, w_lo2 = 3.0e38f;
        if (gp->domain == VGRID_DOMAIN_SPHERE) {
            split_pair(sphere_exit64(gp, P.x, k), th, tl);
            wid = kSphereWall;
            w_lo = __fsub_rd(th, 0x1p-18f * scale);
            w_hi = __fadd_ru(th, 0x1p-18f * scale);
        }
        for (int c = 0; c < 3 && gp->domain != VGRID_DOMAIN_SPHERE; c++) {
            const uint64_t kb = dbits(k[c]);
            if ((kb << 1) == 0) continue;  // k_c = +-0
            const bool up = (kb >> 63) == 0;
            float nh, nl;
            split_pair(__dsub_rn(up ? gp->hi[c] : gp->lo[c], P.x[c]), nh, nl);
            const float kh = p.k_hi[c], kl = p.k_lo[c];
            const float q1 = __fdiv_rn(nh, kh);
            float rem = __fmaf_rn(-q1, kh, nh);
            rem = __fadd_rn(rem, __fmaf_rn(-q1, kl, nl));
            const float q2 = __fdiv_rn(rem, kh);
            float h, l;
            two_sum(q1, q2, h, l);
            if (fp64) {
                const float off = __fmaf_ru(kU, fabsf(h), __fmul_ru(0x1p-36f * scale, __fdiv_ru(1.0f, fabsf(kh))));
                float lo = __fsub_rd(h, off), hi = __fadd_ru(h, off);
                if (!(off < __int_as_float(0x7f800000))) {
                    // k_c is 0 in float32, or so small that the quotient is not a
                    // finite number: no upper bound, and a lower one only where the
                    // moved point is certainly off the wall (then |n| / |k_c|, with
                    // |k_c| below |k_hi| (1 + 2^-22) + 2^-149)
                    const float d = __fsub_rd(__fmul_rd(fabsf(nh), 1.0f - 0x1p-23f), 0x1p-36f * scale);
                    hi = __int_as_float(0x7f800000);
                    lo = d > 0.0f ? __fdiv_rd(d, __fadd_ru(__fmul_ru(fabsf(kh), 1.0f + 0x1p-22f), 0x1p-149f)) : -hi;
                }
                if (lo < w_lo) {
                    w_lo2 = w_lo;
                    w_lo = lo;
                    w_hi = hi;
                } else {
                    w_lo2 = fminf(w_lo2, lo);
                }
            }
            if (h < th || (h == th && l < tl)) {
                th = h;
                tl = l;
                wid = up ? -(2 * c + 2) : -(2 * c + 1);
            }
        }
        if (!(th >= 0.0f) || th > 1.0e38f) {  // start on the boundary facing out (or k = 0)
            th = 0.0f;
            tl = 0.0f;
        } else if (th == 0.0f && tl < 0.0f) {
            tl = 0.0f;
        }
        p.wall = wid;
        p.tmax_hi = th;
        p.tmax_lo = tl;
        float4 *dst = reinterpret_cast<float4 *>(out);
        if (fp64) {
            // a NaN bound (from an infinite one) names no wall either
            const bool one = w_hi < w_lo2 && wid < 0;
            dst[0] = make_float4(__int_as_float(p.cell), __int_as_float(wid), w_lo,
                                 one ? w_hi : __int_as_float(0x7f800000));
            reinterpret_cast<double2 *>(dst)[1] = make_double2(P.x[0], P.x[1]);
            reinterpret_cast<double2 *>(dst)[2] = make_double2(P.x[2], k[0]);
            reinterpret_cast<double2 *>(dst)[3] = make_double2(k[1], k[2]);
        } else {
            const float4 *src = reinterpret_cast<const float4 *>(&p);
            for (int q = 0; q < 4; q++) dst[q] = src[q];
        }
        if (bin) {
            // estimated crossings: (sites per volume)^(1/3) integrated along
            // the in-box segment [0, t_max] with 8 midpoint samples
            int b = 0;
            if (m >= 0 && th > 0.0f) {
                const float dt = th * 0.125f;
                float acc = 0.0f;
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    const float t = (i + 0.5f) * dt;
                    int idx = 0;
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        const float x = __fmaf_rn(t, p.k_hi[c], P.h[c]);
                        const int ic = __float2int_rz(__fmul_rn(__fsub_rn(x, gp->flo_hi[c]), gp->dscale[c]));
                        idx = idx * gp->ddim[c] + max(0, min(ic, gp->ddim[c] - 1));
                    }
                    acc += __ldg(gp->dens + idx);
                }
                const int S = max(1, gp->ospatial), NL = kOrderBins / S;
                const float Q = S == 1 ? 4.0f : 2.0f;  // bins per octave of the estimate
                const int lb = max(0, min(NL - 1, __float2int_rz(Q * __log2f(1.0f + acc * dt))));
                b = lb * S + (S > 1 ? (int)(((int64_t)m * S) / gp->M) : 0);
            }
            bin[w] = (uint8_t)b;
            atomicAdd(&s_hist[b], 1u);
        }
    }
    if (bin) {
        __syncthreads();
        for (int b = threadIdx.x; b < kOrderBins; b += blockDim.x)
            if (s_hist[b]) atomicAdd(&a.hist[b], s_hist[b]);
    }
}

cudaError_t launch_locate(const LocateArgs &a, int prep, int sms, cudaStream_t s) {
    if (a.total <= 0) {
        cudaError_t e = a.queue ? cudaMemsetAsync(a.queue, 0, sizeof(*a.queue), s) : cudaSuccess;
        if (e == cudaSuccess && a.stats) e = cudaMemsetAsync(a.stats, 0, sizeof(*a.stats), s);
        return e;
    }
    // many more blocks than fit: points differ in the records they scan, and the
    // blocks that end early make room (8 / 16 / 32 / 64 per SM and one point per
    // thread took 457 / 452 / 422 / 418 / 435 us for the same points)
    const dim3 g((unsigned)std::min<int64_t>((a.total + 255) / 256, (int64_t)sms * 64));
    switch (prep) {
        case PREP_CELL32: locate_kernel<PREP_CELL32><<<g, 256, 0, s>>>(a); break;
        case PREP_CELL64: locate_kernel<PREP_CELL64><<<g, 256, 0, s>>>(a); break;
        case PREP_FP64: locate_kernel<PREP_FP64><<<g, 256, 0, s>>>(a); break;
        default: locate_kernel<PREP_FP32><<<g, 256, 0, s>>>(a); break;
    }
    count_launches(1);
    return cudaGetLastError();
}

// cursor[b] = number of rays in longer bins (the longest bin goes first)
__global__ void order_scan_kernel(uint32_t *hist) {
    __shared__ uint32_t h[kOrderBins];
    const int b = threadIdx.x;
    h[b] = hist[b];
    __syncthreads();
    uint32_t sum = 0u;
    for (int q = b + 1; q < kOrderBins; q++) sum += h[q];
    hist[kOrderBins + b] = sum;
}

// order[cursor[bin[w]]++] = w in tiles of 2048 rays per block: ranks within
// the tile from shared-memory counters, then one global atomic per bin and
// tile reserves the tile's range (the order inside a bin is arbitrary)
constexpr int kScatterThreads = 256, kScatterPer = 8;
__global__ void __launch_bounds__(kScatterThreads) order_scatter_kernel(const uint8_t *__restrict__ bin,
                                                                        int64_t total, uint32_t *cursor,
                                                                        int32_t *__restrict__ order) {
    __shared__ uint32_t s_cnt[kOrderBins], s_base[kOrderBins];
    const int64_t tile = (int64_t)kScatterThreads * kScatterPer;
    for (int64_t t0 = blockIdx.x * tile; t0 < total; t0 += (int64_t)gridDim.x * tile) {
        if (threadIdx.x < kOrderBins) s_cnt[threadIdx.x] = 0u;
        __syncthreads();
        int b[kScatterPer];
        uint32_t r[kScatterPer];
#pragma unroll
        for (int j = 0; j < kScatterPer; j++) {
            const int64_t w = t0 + (int64_t)j * kScatterThreads + threadIdx.x;
            b[j] = w < total ? (int)__ldg(bin + w) : -1;
            r[j] = b[j] >= 0 ? atomicAdd(&s_cnt[b[j]], 1u) : 0u;
        }
        __syncthreads();
        if (threadIdx.x < kOrderBins)
            s_base[threadIdx.x] = s_cnt[threadIdx.x] ? atomicAdd(&cursor[threadIdx.x], s_cnt[threadIdx.x]) : 0u;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kScatterPer; j++) {
            const int64_t w = t0 + (int64_t)j * kScatterThreads + threadIdx.x;
            if (b[j] >= 0) order[s_base[b[j]] + r[j]] = (int32_t)w;
        }
        __syncthreads();
    }
}

cudaError_t launch_order(const RayOrder &ord, int64_t total, int sms, cudaStream_t s) {
    if (total <= 0) return cudaSuccess;
    order_scan_kernel<<<1, kOrderBins, 0, s>>>(ord.hist);
    count_launches(1);
    const int64_t tile = (int64_t)kScatterThreads * kScatterPer;
    int64_t blocks = (total + tile - 1) / tile;
    blocks = blocks < (int64_t)sms * 8 ? blocks : (int64_t)sms * 8;
    order_scatter_kernel<<<(unsigned)blocks, kScatterThreads, 0, s>>>(ord.bin, total, ord.hist + kOrderBins,
                                                                     ord.order);
    count_launches(1);
    return cudaGetLastError();
}

// rho (caller order) into the headers of both forms of the cell blocks
__global__ void permute_density_kernel(const float *__restrict__ rho_caller, const int32_t *__restrict__ perm,
                                       const float4 *__restrict__ site, int64_t M, float4 *cells, float4 *rel) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const int f = __float_as_int(__ldg(&site[i]).w);
        const float v = __ldg(&rho_caller[__ldg(&perm[i])]);
        float4 *h1 = rel + f + 1;
        h1->y = v;
        cells[__float_as_int(h1->w)].z = v;
    }
}

cudaError_t launch_permute_density(const float *rho_caller, const int32_t *perm, const float4 *site, int64_t M,
                                   float4 *cells, float4 *rel, cudaStream_t s) {
    if (M <= 0) return cudaSuccess;
    int64_t blocks = (M + 255) / 256;
    if (blocks > 65535) blocks = 65535;
    permute_density_kernel<<<(unsigned)blocks, 256, 0, s>>>(rho_caller, perm, site, M, cells, rel);
    count_launches(1);
    return cudaGetLastError();
}

// Rays that start outside the box move to where they enter it: the slab
// test gives the parameter interval [t_in, t_out] in which the line is
// inside every slab; a ray with t_in <= t_out and t_out >= 0 starts at
// r0 + max(t_in, 0) k, clamped into the closed box against rounding. Rays
// inside are copied unchanged, rays that miss keep their outside origin.
// In a spherical domain a ray outside the ball (q = o.o - R^2 > 0, o = r0 -
// c) that meets it ahead (b = k.o < 0, b^2 - q >= 0) starts epsilon past the
// smaller root, q / (sqrt(b^2 - q) - b) + epsilon (no digits cancel), every
// operation rounded to nearest in this order.
__global__ void enter_kernel(const double *__restrict__ origin, const double *__restrict__ dir, int64_t N,
                             const GridDev *gp, double *__restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        double r[3], k[3];
        bool in = true;
        for (int c = 0; c < 3; c++) {
            r[c] = origin[3 * i + c];
            k[c] = dir[3 * i + c];
            in = in && r[c] >= gp->lo[c] && r[c] <= gp->hi[c];
        }
        if (gp->domain == VGRID_DOMAIN_SPHERE) {
            double o[3];
            for (int c = 0; c < 3; c++) o[c] = __dsub_rn(r[c], gp->sph[c]);
            const double q = __dsub_rn(__dadd_rn(__dadd_rn(__dmul_rn(o[0], o[0]), __dmul_rn(o[1], o[1])),
                                                 __dmul_rn(o[2], o[2])),
                                       __dmul_rn(gp->sph[3], gp->sph[3]));
            if (q > 0.0) {
                const double b = __dadd_rn(__dadd_rn(__dmul_rn(k[0], o[0]), __dmul_rn(k[1], o[1])), __dmul_rn(k[2], o[2]));
                const double disc = __dsub_rn(__dmul_rn(b, b), q);
                if (b < 0.0 && disc >= 0.0) {
                    const double t = __dadd_rn(__ddiv_rn(q, __dsub_rn(__dsqrt_rn(disc), b)), gp->eps64);
                    for (int c = 0; c < 3; c++) r[c] = __dadd_rn(r[c], __dmul_rn(t, k[c]));
                }
            }
        } else if (!in) {
            double t_in = -1e300, t_out = 1e300;
            bool miss = false;
            for (int c = 0; c < 3; c++) {
                if (k[c] != 0.0) {
                    const double t1 = (gp->lo[c] - r[c]) / k[c], t2 = (gp->hi[c] - r[c]) / k[c];
                    t_in = fmax(t_in, fmin(t1, t2));
                    t_out = fmin(t_out, fmax(t1, t2));
                } else if (r[c] < gp->lo[c] || r[c] > gp->hi[c]) {
                    miss = true;
                }
            }
            if (!miss && t_in <= t_out && t_out >= 0.0) {
                const double t = fmax(t_in, 0.0);
                for (int c = 0; c < 3; c++) r[c] = fmin(fmax(__fma_rn(t, k[c], r[c]), gp->lo[c]), gp->hi[c]);
            }
        }
        for (int c = 0; c < 3; c++) out[3 * i + c] = r[c];
    }
}

cudaError_t launch_enter(const double *origin, const double *dir, int64_t N, const GridDev *gp, double *out, int sms,
                         cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    int64_t blocks = (N + 255) / 256;
    blocks = blocks < (int64_t)sms * 16 ? blocks : (int64_t)sms * 16;
    enter_kernel<<<(unsigned)blocks, 256, 0, s>>>(origin, dir, N, gp, out);
    count_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// exclusive prefix sum over int64 (three passes: tiles, tile totals, fix-up)
// ---------------------------------------------------------------------------

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int64_t kScanTile = (int64_t)kScanThreads * kScanItems;

__device__ __forceinline__ int64_t block_exclusive_scan(int64_t v, int64_t *warp_sums, int64_t &block_total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int64_t w = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_sums[lane] = w;  // inclusive over warps
    }
    __syncthreads();
    block_total = warp_sums[(blockDim.x >> 5) - 1];
    const int64_t before = wid > 0 ? warp_sums[wid - 1] : 0;
    const int64_t r = before + x - v;
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kScanThreads) scan_tiles_kernel(int64_t *data, int64_t n, int64_t *tile_sums) {
    __shared__ int64_t ws[32];
    const int64_t base = blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    int64_t v[kScanItems];
    int64_t sum = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        v[i] = base + i < n ? data[base + i] : 0;
        sum += v[i];
    }
    int64_t total;
    int64_t run = block_exclusive_scan(sum, ws, total);
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        if (base + i < n) data[base + i] = run;
        run += v[i];
    }
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) scan_sums_kernel(int64_t *tile_sums, int64_t ntiles, int64_t *out_total) {
    __shared__ int64_t ws[32];
    int64_t carry = 0;
    for (int64_t b = 0; b < ntiles; b += kScanThreads) {
        const int64_t i = b + threadIdx.x;
        const int64_t v = i < ntiles ? tile_sums[i] : 0;
        int64_t total;
        const int64_t ex = block_exclusive_scan(v, ws, total);
        if (i < ntiles) tile_sums[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) *out_total = carry;
}

__global__ void __launch_bounds__(kScanThreads) scan_fix_kernel(int64_t *data, int64_t n, const int64_t *tile_sums) {
    const int64_t add = tile_sums[blockIdx.x];
    const int64_t base = blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
#pragma unroll
    for (int i = 0; i < kScanItems; i++)
        if (base + i < n) data[base + i] += add;
}

// Offsets of the rays' segments and of their chunks (ceil(n / kSegChunk)), both
// scans in one pass over the counts: three kernels instead of seven, and the
// counts are read once.
__global__ void __launch_bounds__(kScanThreads) ray_scan_tiles_kernel(int64_t *off, int64_t n, int64_t *coff,
                                                                     longlong2 *tile_sums) {
    __shared__ int64_t ws[32];
    const int64_t base = blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    int64_t v[kScanItems], sum = 0, csum = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        v[i] = base + i < n ? off[base + i] : 0;
        sum += v[i];
        csum += (v[i] + kSegChunk - 1) / kSegChunk;
    }
    int64_t total, ctotal;
    int64_t run = block_exclusive_scan(sum, ws, total), crun = block_exclusive_scan(csum, ws, ctotal);
#pragma unroll
    for (int i = 0; i < kScanItems; i++) {
        if (base + i < n) {
            off[base + i] = run;
            coff[base + i] = crun;
        }
        run += v[i];
        crun += (v[i] + kSegChunk - 1) / kSegChunk;
    }
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = make_longlong2(total, ctotal);
}

__global__ void __launch_bounds__(kScanThreads) ray_scan_sums_kernel(longlong2 *tile_sums, int64_t ntiles, int64_t *off_n,
                                                                    int64_t *coff_n) {
    __shared__ int64_t ws[32];
    int64_t carry = 0, ccarry = 0;
    for (int64_t b = 0; b < ntiles; b += kScanThreads) {
        const int64_t i = b + threadIdx.x;
        const longlong2 v = i < ntiles ? tile_sums[i] : make_longlong2(0, 0);
        int64_t total, ctotal;
        const int64_t ex = block_exclusive_scan(v.x, ws, total), cex = block_exclusive_scan(v.y, ws, ctotal);
        if (i < ntiles) tile_sums[i] = make_longlong2(carry + ex, ccarry + cex);
        carry += total;
        ccarry += ctotal;
    }
    if (threadIdx.x == 0) {
        *off_n = carry;
        *coff_n = ccarry;
    }
}

__global__ void __launch_bounds__(kScanThreads) ray_scan_fix_kernel(int64_t *off, int64_t n, int64_t *coff,
                                                                   const longlong2 *tile_sums) {
    const longlong2 add = tile_sums[blockIdx.x];
    const int64_t base = blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
#pragma unroll
    for (int i = 0; i < kScanItems; i++)
        if (base + i < n) {
            off[base + i] += add.x;
            coff[base + i] += add.y;
        }
}

// Chunked segments -> CSR, in the order of the destination so that the
// stores are coalesced: each used chunk c of ray r at position k is entered as
// inv[coff[r] + k] = c; then kSegChunk threads per destination chunk copy its
// slots to the ray's offset plus kSegChunk * k. The number of chunks the
// traversal took and the total are read on the device: when the total
// exceeds the caller's capacity (some chunks were never stored) both do
// nothing, and only the offsets go back. (Entering (c, r) in inv, so that a
// chunk's slots and its ray's offsets load side by side, and two slots per
// thread took 47 + 148 us for 28.7 10^6 segments instead of 36 + 133: the
// inversion's scattered writes double and the copy's are 8 bytes apart.)
__global__ void chunk_invert_kernel(const int2 *meta, const unsigned long long *cursor, int64_t chunk_cap,
                                    const int64_t *off, int64_t N, int64_t cap, const int64_t *coff, int32_t *inv) {
    if (__ldg(off + N) > cap) return;
    const int64_t nchunks = min((int64_t)*cursor, chunk_cap);
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nchunks;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int2 m = __ldg(meta + c);
        if (m.x >= 0) inv[__ldg(coff + m.x) + m.y] = (int32_t)c;  // -1: handed to a warp, not used
    }
}

template <bool FP64>
__global__ void __launch_bounds__(256) compact_segments_kernel(const int64_t *off, const int64_t *coff, int64_t N,
                                                               int64_t cap, const int32_t *inv, const int2 *meta,
                                                               const void *slots, int32_t *cell, void *len) {
    if (__ldg(off + N) > cap) return;
    const int64_t nd = __ldg(coff + N);  // destination chunks
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nd * kSegChunk; t += stride) {
        const int32_t c = __ldg(inv + t / kSegChunk);
        const int2 m = __ldg(meta + c);
        const int64_t o = __ldg(off + m.x), n = __ldg(off + m.x + 1) - o;
        const int64_t j = (int64_t)m.y * kSegChunk + (t & (kSegChunk - 1));
        if (j >= n) continue;
        const int64_t at = (int64_t)c * kSegChunk + (t & (kSegChunk - 1));
        if (FP64) {
            const int4 v = __ldcs(reinterpret_cast<const int4 *>(slots) + at);
            cell[o + j] = v.x;
            reinterpret_cast<double *>(len)[o + j] = __hiloint2double(v.w, v.z);
        } else {
            const int2 v = __ldcs(reinterpret_cast<const int2 *>(slots) + at);
            cell[o + j] = v.x;
            reinterpret_cast<float *>(len)[o + j] = __int_as_float(v.y);
        }
    }
}

static int grid_for(int64_t threads, int sms) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((threads + 255) / 256, (int64_t)sms * 8));
}

int64_t segment_tmp_elems(int64_t n) { return 2 * scan_tmp_elems(n); }

cudaError_t launch_segment_lists(int64_t *off, int64_t N, int64_t chunk_cap, const unsigned long long *cursor,
                                 const int2 *meta, const void *slots, bool fp64, int64_t cap, int64_t *coff,
                                 int64_t *scan_tmp, int32_t *inv, int32_t *cell, void *len, int sms, cudaStream_t s) {
    if (N <= 0) return cudaMemsetAsync(off, 0, sizeof(int64_t), s);
    const int64_t tiles = (N + kScanTile - 1) / kScanTile;
    longlong2 *const sums = reinterpret_cast<longlong2 *>(scan_tmp);
    ray_scan_tiles_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(off, N, coff, sums);
    ray_scan_sums_kernel<<<1, kScanThreads, 0, s>>>(sums, tiles, off + N, coff + N);
    ray_scan_fix_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(off, N, coff, sums);
    count_launches(3);
    if (chunk_cap <= 0 || !cell || !len) return cudaGetLastError();
    chunk_invert_kernel<<<grid_for(chunk_cap, sms), 256, 0, s>>>(meta, cursor, chunk_cap, off, N, cap, coff, inv);
    // destination chunks: coff[N] (read on the device), at most chunk_cap
    if (fp64)
        compact_segments_kernel<true><<<grid_for(chunk_cap * kSegChunk, sms), 256, 0, s>>>(off, coff, N, cap, inv,
                                                                                           meta, slots, cell, len);
    else
        compact_segments_kernel<false><<<grid_for(chunk_cap * kSegChunk, sms), 256, 0, s>>>(off, coff, N, cap, inv,
                                                                                            meta, slots, cell, len);
    count_launches(2);
    return cudaGetLastError();
}

// 8 lanes per ray striding over its segments (coalesced reads of the
// lists); the term is (dL/dtau_r kappa) l, as the traversal's adjoint forms it
__global__ void segments_grad_kernel(const int64_t *off, const int32_t *cell, const float *len, int64_t N,
                                     const float *g, float kappa, float *out) {
    const int i = threadIdx.x & 7;
    const int64_t groups = (int64_t)gridDim.x * blockDim.x / 8;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 8; r < N; r += groups) {
        const float gk = __ldg(g + r) * kappa;
        const int64_t a = __ldg(off + r), b = __ldg(off + r + 1);
        for (int64_t k = a + i; k < b; k += 8) atomicAdd(out + __ldg(cell + k), gk * __ldg(len + k));
    }
}

cudaError_t launch_segments_grad(const int64_t *off, const int32_t *cell, const float *len, int64_t N, const float *g,
                                 float kappa, float *out, int sms, cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((N * 8 + 255) / 256, (int64_t)sms * 8));
    segments_grad_kernel<<<blocks, 256, 0, s>>>(off, cell, len, N, g, kappa, out);
    count_launches(1);
    return cudaGetLastError();
}

int64_t scan_tmp_elems(int64_t n) { return (n + kScanTile - 1) / kScanTile + 1; }

cudaError_t launch_exclusive_scan(int64_t *data, int64_t n, int64_t *tmp, cudaStream_t s) {
    const int64_t tiles = (n + kScanTile - 1) / kScanTile;
    if (tiles == 0) {
        return cudaMemsetAsync(data, 0, sizeof(int64_t), s);
    }
    scan_tiles_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(data, n, tmp);
    count_launches(1);
    scan_sums_kernel<<<1, kScanThreads, 0, s>>>(tmp, tiles, data + n);
    count_launches(1);
    scan_fix_kernel<<<(unsigned)tiles, kScanThreads, 0, s>>>(data, n, tmp);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace vg
