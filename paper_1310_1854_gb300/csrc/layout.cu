// Device arrays of a grid, built on the device from the cells (neighbour
// lists and bounding boxes): the cell blocks of both forms, the block lists of
// C(r) (Sect. 2.3) and the coarse density grid of the ray order.
//
// The host used to write these arrays (about 0.9 KB per cell) and copy them in:
// 25 ms of the 72 ms that a grid of 10^5 sites with GPU-built cells takes, most
// of 0.27 s of the 0.41 s at 10^6 sites. All of it is gathers and scatters per
// cell or per block, one warp each here.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"
#include "kernels.h"

namespace vg {
namespace {

constexpr int kWarps = 8;               // warps per block of the kernels below
constexpr int kMaxNeighbours = 4096;    // a cell with more has its records ordered on the host
constexpr int kMaxList = 256;           // a block list with more entries is a thread block's work, not a warp's
constexpr int kLongThreads = 256;

__device__ __forceinline__ int64_t warp_index() {
    return ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
}
__device__ __forceinline__ int64_t warp_count() { return ((int64_t)gridDim.x * blockDim.x) >> 5; }

__device__ __forceinline__ float nan_f() { return __int_as_float(0x7fc00000); }

// (squared distance, id) as one number that orders like the pair
__device__ __forceinline__ unsigned long long near_key(float d2, int id) {
    return ((unsigned long long)__float_as_uint(d2) << 32) | (unsigned)id;
}

// |unit n|^2 with the operations of the search's early stop
__device__ __forceinline__ float norm2(float unit, float x, float y, float z) {
    x = __fmul_rn(unit, x);
    y = __fmul_rn(unit, y);
    z = __fmul_rn(unit, z);
    return __fmaf_rn(z, z, __fmaf_rn(y, y, __fmul_rn(x, x)));
}

// entries of a cell's two blocks: 1 + neighbours and walls; 2 + cell
// neighbours, at least four and an even count
__global__ void cell_sizes_kernel(const int64_t *off, const int32_t *idx, int64_t M, int64_t *a, int64_t *f) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = off[i], e = off[i + 1];
        int n = 0;
        for (int64_t q = b; q < e; q++) n += idx[q] >= 0;
        a[i] = 1 + (e - b);
        f[i] = 2 + max(4, (n + 1) & ~1);
    }
}

__global__ void sites_kernel(const float4 *site, const int64_t *foffs, int64_t M, float4 *out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 q = site[i];
        out[i] = make_float4(q.x, q.y, q.z, __int_as_float((int)foffs[i]));
    }
}

// One warp per cell: its absolute block (records in list order) and its
// relative block (records by |p_j - p_i|^2, ties by cell, each placed at its
// rank). Cells with more neighbours than kMaxNeighbours keep the list order
// there and are counted in *big.
__global__ void __launch_bounds__(32 * kWarps) cell_blocks_kernel(const float4 *site, const int32_t *perm,
                                                                  const int64_t *off, const int32_t *idx, int64_t M,
                                                                  const int64_t *aoffs, const int64_t *foffs,
                                                                  float unit, float4 *cells, float4 *rel, int *big) {
    const int lane = threadIdx.x & 31;
    for (int64_t i = warp_index(); i < M; i += warp_count()) {
        const int64_t b = off[i];
        const int n = (int)(off[i + 1] - b);
        const int64_t A = aoffs[i], F = foffs[i];
        const int c4 = (int)(foffs[i + 1] - F) - 2;
        const float4 p = site[i];
        const bool sort = n <= kMaxNeighbours;
        double n1max = 0.0;
        int ncell = 0;
        for (int q0 = 0; q0 < n; q0 += 32) {
            const int q = q0 + lane;
            const int j = q < n ? idx[b + q] : -1;
            const bool cell = j >= 0;
            const unsigned cm = __ballot_sync(0xffffffffu, cell);
            float4 r = make_float4(0.f, 0.f, 0.f, __int_as_float(j));
            float4 d = r;
            if (cell) {
                const float4 s = site[j];
                r = make_float4(s.x, s.y, s.z, __int_as_float((int)aoffs[j]));
                // one float32 rounding, as a subtraction in the traversal would be
                d = make_float4(__fsub_rn(s.x, p.x), __fsub_rn(s.y, p.y), __fsub_rn(s.z, p.z),
                                __int_as_float((int)foffs[j]));
                n1max = fmax(n1max, fabs((double)d.x) + fabs((double)d.y) + fabs((double)d.z));
            }
            if (q < n) cells[A + 1 + q] = r;
            int rank = ncell + __popc(cm & ((1u << lane) - 1u));
            if (sort) {
                const unsigned long long key = near_key(norm2(unit, d.x, d.y, d.z), j);
                rank = 0;
                for (int t = 0; t < n; t++) {
                    const int k = idx[b + t];
                    if (k < 0) continue;
                    const float4 s = site[k];
                    const float x = __fsub_rn(s.x, p.x), y = __fsub_rn(s.y, p.y), z = __fsub_rn(s.z, p.z);
                    rank += near_key(norm2(unit, x, y, z), k) < key;
                }
            }
            if (cell) rel[F + 2 + rank] = d;
            ncell += __popc(cm);
        }
        for (int o = 16; o; o >>= 1) n1max = fmax(n1max, __shfl_xor_sync(0xffffffffu, n1max, o));
        for (int k = ncell + lane; k < c4; k += 32)
            rel[F + 2 + k] = make_float4(nan_f(), nan_f(), nan_f(), __int_as_float(-8));
        if (lane == 0) {
            // rho is 1 until set_density
            cells[A] = make_float4(__int_as_float(perm[i]), __int_as_float(n), 1.0f, __int_as_float((int)F));
            rel[F] = make_float4(p.x, p.y, p.z, __int_as_float(c4));
            rel[F + 1] = make_float4(__int_as_float(perm[i]), 1.0f, __double2float_ru(n1max * (1.0 + 1e-6)),
                                     __int_as_float((int)A));
            if (!sort) atomicAdd(big, 1);
        }
    }
}

// the entries past the last block, for the last block's reads
__global__ void tail_kernel(float4 *cells, int64_t na, float4 *rel, int64_t nf) {
    const int t = threadIdx.x;
    cells[na + t] = make_float4(0.f, 0.f, 0.f, __int_as_float(-8));
    rel[nf + t] = make_float4(nan_f(), nan_f(), nan_f(), __int_as_float(-8));
}

struct BlockDev {
    double lo[3], ext[3], pad;
    int dim[3];
    float flo[3], fbw[3];
};

// A warp takes five cells at a time, over the blocks that each one's bounding
// box, padded, overlaps. FILL: enter the cell's record in each (anywhere in the
// list, at the block's cursor); otherwise count them. The six ends of the five
// boxes are one lane's each: a warp pays a float64 division in full whether one
// lane or all need it, and with every lane forming all six for one cell at a time
// that bound both passes (10^5 cells 514 and 526 us, 10^6 5.0 and 5.1 ms; 31 and
// 97 us, 0.27 and 1.2 ms now).
constexpr int kBoxCells = 5;

template <bool FILL>
__global__ void __launch_bounds__(32 * kWarps) block_lists_kernel(const double *bbox, int64_t M, BlockDev g,
                                                                  const float4 *site, const int32_t *boff,
                                                                  unsigned *cnt, float4 *rec) {
    const int lane = threadIdx.x & 31;
    const int s = lane % 6, x = s % 3;  // end s of the box of cell lane / 6, along axis x
    const double lo = x == 0 ? g.lo[0] : x == 1 ? g.lo[1] : g.lo[2];
    const double ext = x == 0 ? g.ext[0] : x == 1 ? g.ext[1] : g.ext[2];
    const int dim = x == 0 ? g.dim[0] : x == 1 ? g.dim[1] : g.dim[2];
    for (int64_t m0 = warp_index() * kBoxCells; m0 < M; m0 += warp_count() * kBoxCells) {
        const int cells = (int)min(M - m0, (int64_t)kBoxCells);
        int v = 0;
        if (lane < 6 * cells) {
            const double e = bbox[6 * m0 + lane];
            const double w = floor(((s < 3 ? e - g.pad : e + g.pad) - lo) / ext * dim);
            v = s < 3 ? (int)fmax(0.0, w) : (int)fmin((double)dim - 1.0, w);
        }
        for (int c = 0; c < cells; c++) {
            int a[3], b[3];
            for (int q = 0; q < 3; q++) {
                a[q] = __shfl_sync(0xffffffffu, v, 6 * c + q);
                b[q] = __shfl_sync(0xffffffffu, v, 6 * c + 3 + q);
            }
            // at most 1024 blocks per axis
            const unsigned nj = b[1] - a[1] + 1, nk = b[2] - a[2] + 1, n = (b[0] - a[0] + 1) * nj * nk;
            float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
            if (FILL) {
                const float4 p = site[m0 + c];
                r = make_float4(p.x, p.y, p.z, __int_as_float((int)(m0 + c)));
            }
            for (unsigned t = lane; t < n; t += 32) {
                const unsigned i = a[0] + t / (nj * nk), j = a[1] + t / nk % nj, k = a[2] + t % nk;
                const unsigned q = (i * g.dim[1] + j) * g.dim[2] + k;
                const unsigned at = atomicAdd(cnt + q, 1u);
                if (FILL) rec[(int64_t)boff[q] + at] = r;
            }
        }
    }
}

// list lengths rounded up to even, as int64 for the scan; *odd counts the odd ones
__global__ void even_kernel(const unsigned *cnt, int64_t K, int64_t *off, unsigned *odd) {
    unsigned n = 0;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < K; q += (int64_t)gridDim.x * blockDim.x) {
        off[q] = ((int64_t)cnt[q] + 1) & ~(int64_t)1;
        n += cnt[q] & 1u;
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(odd, n);
}

__global__ void narrow_kernel(const int64_t *off, int64_t n, int32_t *out) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        out[q] = (int32_t)off[q];
}

// the key of a record in the list of block q
struct BlockKey {
    float cen[3];
    __device__ BlockKey(const BlockDev &g, int64_t q) {
        const int64_t bk[3] = {q / ((int64_t)g.dim[1] * g.dim[2]), (q / g.dim[2]) % g.dim[1], q % g.dim[2]};
        for (int c = 0; c < 3; c++)
            cen[c] = __fadd_rn(g.flo[c], __fmul_rn(__fadd_rn((float)bk[c], 0.5f), g.fbw[c]));
    }
    __device__ unsigned long long operator()(float4 r) const {
        const float x = __fsub_rn(r.x, cen[0]), y = __fsub_rn(r.y, cen[1]), z = __fsub_rn(r.z, cen[2]);
        return near_key(__fmaf_rn(z, z, __fmaf_rn(y, y, __fmul_rn(x, x))), __float_as_int(r.w));
    }
};

// Order every list by the sites' squared distance from its block's centre
// (float32, computed as the start-cell search computes the centre; its margin
// of 16u covers this order), ties by cell, and pad it to an even length with
// a NaN record. One warp per block: a record's rank is the number of smaller
// keys, so that a list is ordered in place after one read. Lists longer than
// kMaxList are noted in `big` (room for K), unordered.
__global__ void __launch_bounds__(32 * kWarps) order_lists_kernel(const int32_t *boff, const unsigned *cnt, int64_t K,
                                                                  BlockDev g, float4 *rec, int64_t *big,
                                                                  unsigned *nbig) {
    __shared__ unsigned long long s_key[kWarps][kMaxList];
    __shared__ float s_rec[kWarps][kMaxList][3];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t q = warp_index(); q < K; q += warp_count()) {
        const int n = (int)cnt[q];
        float4 *const list = rec + boff[q];
        if (lane == 0 && (n & 1)) list[n] = make_float4(nan_f(), nan_f(), nan_f(), __int_as_float(-1));
        if (n < 2) continue;
        const BlockKey key_of(g, q);
        if (n <= 32) {
            float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
            unsigned long long key = ~0ull;
            if (lane < n) {
                r = list[lane];
                key = key_of(r);
            }
            int rank = 0;
            for (int t = 0; t < n; t++) rank += __shfl_sync(0xffffffffu, key, t) < key;
            __syncwarp();
            if (lane < n) list[rank] = r;
        } else if (n <= kMaxList) {
            for (int i = lane; i < n; i += 32) {
                const float4 r = list[i];
                s_key[w][i] = key_of(r);
                s_rec[w][i][0] = r.x;
                s_rec[w][i][1] = r.y;
                s_rec[w][i][2] = r.z;
            }
            __syncwarp();
            for (int i = lane; i < n; i += 32) {
                const unsigned long long key = s_key[w][i];
                int rank = 0;
                for (int t = 0; t < n; t++) rank += s_key[w][t] < key;
                list[rank] = make_float4(s_rec[w][i][0], s_rec[w][i][1], s_rec[w][i][2],
                                         __int_as_float((int)(unsigned)key));
            }
            __syncwarp();
        } else if (lane == 0) {
            big[atomicAdd(nbig, 1u)] = q;
        }
    }
}

// The lists noted above, one thread block each: a bitonic network in place (the
// blocks' barriers order their own reads and writes), in the form that always
// moves the smaller key down, so that entries past the end count as the largest
// keys and stay there. Few blocks per site make them, or sites crowded into one
// block: 10^6 uniform sites at 0.003 blocks per site have 2744 lists of 610, which
// took the host 154 ms, one after the other with four copies each; 1 ms now, and
// the whole grid 0.164 s instead of 0.317.
__global__ void __launch_bounds__(kLongThreads) order_long_lists_kernel(const int64_t *big, unsigned nbig,
                                                                       const int32_t *boff, const unsigned *cnt,
                                                                       BlockDev g, float4 *rec) {
    for (unsigned l = blockIdx.x; l < nbig; l += gridDim.x) {
        const int64_t q = big[l];
        const unsigned n = cnt[q];
        float4 *const list = rec + boff[q];
        const BlockKey key_of(g, q);
        auto in_order = [&](unsigned i, unsigned k) {
            if (k >= n) return;
            const float4 a = list[i], b = list[k];
            if (key_of(b) < key_of(a)) {
                list[i] = b;
                list[k] = a;
            }
        };
        unsigned half = 1;  // half of the smallest power of two that holds the list
        while (2 * half < n) half *= 2;
        for (unsigned k = 2; k <= 2 * half; k *= 2) {
            for (unsigned t = threadIdx.x; t < half; t += kLongThreads) {
                const unsigned r = t & (k / 2 - 1), base = 2 * (t - r);
                in_order(base + r, base + k - 1 - r);
            }
            __syncthreads();
            for (unsigned j = k / 4; j > 0; j /= 2) {
                for (unsigned t = threadIdx.x; t < half; t += kLongThreads) {
                    const unsigned r = t & (j - 1), i = 2 * (t - r) + r;
                    in_order(i, i + j);
                }
                __syncthreads();
            }
        }
    }
}

__global__ void density_count_kernel(const float4 *site, int64_t M, BlockDev g, unsigned *cnt) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 s = site[i];
        const double x[3] = {(double)s.x, (double)s.y, (double)s.z};
        int64_t at = 0;
        for (int c = 0; c < 3; c++) {
            const double f = (x[c] - g.lo[c]) / g.ext[c] * g.dim[c];
            at = at * g.dim[c] + min(max((int64_t)f, (int64_t)0), (int64_t)g.dim[c] - 1);
        }
        atomicAdd(cnt + at, 1u);
    }
}

__global__ void density_kernel(const unsigned *cnt, int64_t n, double vol, float *dens) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dens[i] = (float)cbrt(fmax(0.25, (double)cnt[i]) / vol);
}

int blocks_for(int64_t items, int per_block, int sms) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((items + per_block - 1) / per_block, (int64_t)sms * 32));
}

// device memory freed when the scope ends, unless taken
struct Temp {
    std::vector<void *> p;
    ~Temp() {
        for (void *q : p)
            if (q) cudaFree(q);
    }
    template <class T>
    cudaError_t get(T **out, int64_t n) {
        *out = nullptr;
        void *q = nullptr;
        const cudaError_t e = cudaMalloc(&q, sizeof(T) * (size_t)std::max<int64_t>(n, 1));
        if (e == cudaSuccess) {
            p.push_back(q);
            *out = static_cast<T *>(q);
        } else {
            cudaGetLastError();
        }
        return e;
    }
    void take(void *q) { std::replace(p.begin(), p.end(), q, (void *)nullptr); }
};

}  // namespace

int build_layout(const LayoutIn &in, LayoutOut &out, std::string &err) {
    const int64_t M = in.M;
    Temp tmp, keep;
    cudaError_t e = cudaSuccess;
    auto bad = [&](const char *what) {
        err = std::string(what) + ": " + cudaGetErrorString(e);
        return e == cudaErrorMemoryAllocation ? LAYOUT_NOMEM : LAYOUT_CUDA;
    };
#define VG_TRY(call) \
    if ((e = (call)) != cudaSuccess) return bad(#call)
    auto t0 = std::chrono::steady_clock::now();
    auto lap = [&]() {
        const auto now = std::chrono::steady_clock::now();
        const double d = std::chrono::duration<double>(now - t0).count();
        t0 = now;
        return d;
    };
    // inputs on the device
    float4 *s4 = nullptr;
    VG_TRY(tmp.get(&s4, M));
    VG_TRY(cudaMemcpy(s4, in.site4, sizeof(float4) * M, cudaMemcpyHostToDevice));
    VG_TRY(keep.get(&out.perm, M));
    VG_TRY(cudaMemcpy(out.perm, in.perm, sizeof(int32_t) * M, cudaMemcpyHostToDevice));
    const int64_t nnz = in.off[M];
    const int64_t *off = in.d_off;
    const int32_t *idx = in.d_idx;
    const double *bbox = in.d_bbox;
    if (!off || !idx) {
        int64_t *o = nullptr;
        int32_t *x = nullptr;
        VG_TRY(tmp.get(&o, M + 1));
        VG_TRY(tmp.get(&x, nnz));
        VG_TRY(cudaMemcpy(o, in.off, sizeof(int64_t) * (M + 1), cudaMemcpyHostToDevice));
        VG_TRY(cudaMemcpy(x, in.idx, sizeof(int32_t) * nnz, cudaMemcpyHostToDevice));
        off = o;
        idx = x;
    }
    if (!bbox) {
        double *b = nullptr;
        VG_TRY(tmp.get(&b, 6 * M));
        VG_TRY(cudaMemcpy(b, in.bbox, sizeof(double) * 6 * M, cudaMemcpyHostToDevice));
        bbox = b;
    }
    out.seconds[0] = lap();
    // block lists
    int64_t *scan = nullptr;
    BlockDev g;
    double ext[3], maxabs = 0.0;
    for (int c = 0; c < 3; c++) {
        ext[c] = in.box[3 + c] - in.box[c];
        g.lo[c] = in.box[c];
        g.ext[c] = ext[c];
        g.dim[c] = in.bdim[c];
        g.flo[c] = (float)in.box[c];
        g.fbw[c] = (float)(ext[c] / in.bdim[c]);
    }
    for (int c = 0; c < 6; c++) maxabs = std::max(maxabs, std::fabs(in.box[c]));
    g.pad = 1e-6 * std::sqrt(ext[0] * ext[0] + ext[1] * ext[1] + ext[2] * ext[2]) + 1e-13 * maxabs;
    const int64_t K = (int64_t)in.bdim[0] * in.bdim[1] * in.bdim[2];
    VG_TRY(tmp.get(&scan, scan_tmp_elems(std::max(K, M))));
    unsigned *cnt = nullptr, *nbig = nullptr;
    int64_t *boff = nullptr;
    VG_TRY(tmp.get(&cnt, K));
    VG_TRY(tmp.get(&boff, K + 1));
    VG_TRY(tmp.get(&nbig, 3));  // long lists, cells with many neighbours, odd lists
    VG_TRY(cudaMemset(cnt, 0, sizeof(unsigned) * K));
    VG_TRY(cudaMemset(nbig, 0, 3 * sizeof(unsigned)));
    const int wb = 32 * kWarps;
    block_lists_kernel<false><<<blocks_for(M, kBoxCells * kWarps, in.sms), wb>>>(bbox, M, g, nullptr, nullptr, cnt, nullptr);
    even_kernel<<<blocks_for(K, 256, in.sms), 256>>>(cnt, K, boff, nbig + 2);
    VG_TRY(launch_exclusive_scan(boff, K, scan, 0));
    int64_t total = 0;
    VG_TRY(cudaMemcpy(&total, boff + K, sizeof(int64_t), cudaMemcpyDeviceToHost));
    if (total + K + 2 >= ((int64_t)1 << 31)) {
        err = "block lists exceed 2^31 entries; lower blocks_per_site";
        return LAYOUT_NOMEM;
    }
    VG_TRY(keep.get(&out.blk_off, K + 1));
    VG_TRY(keep.get(&out.blk_rec, total + 2));
    narrow_kernel<<<blocks_for(K + 1, 256, in.sms), 256>>>(boff, K + 1, out.blk_off);
    VG_TRY(cudaMemset(cnt, 0, sizeof(unsigned) * K));
    block_lists_kernel<true><<<blocks_for(M, kBoxCells * kWarps, in.sms), wb>>>(bbox, M, g, s4, out.blk_off, cnt, out.blk_rec);
    // (the scanned offsets are in out.blk_off by now: their buffer holds the long lists)
    order_lists_kernel<<<blocks_for(K, kWarps, in.sms), wb>>>(out.blk_off, cnt, K, g, out.blk_rec, boff, nbig);
    count_launches(5);
    unsigned nlong = 0;
    VG_TRY(cudaMemcpy(&nlong, nbig, sizeof(nlong), cudaMemcpyDeviceToHost));
    if (nlong) {
        order_long_lists_kernel<<<std::min(nlong, (unsigned)in.sms * 8), kLongThreads>>>(boff, nlong, out.blk_off, cnt, g,
                                                                                        out.blk_rec);
        count_launches(1);
    }
    // the two records past the last list
    const float fnan = std::nanf("");
    float4 pad2[2];
    for (float4 &r : pad2) {
        r = make_float4(fnan, fnan, fnan, 0.f);
        const int32_t none = -1;
        std::copy(reinterpret_cast<const char *>(&none), reinterpret_cast<const char *>(&none) + 4,
                  reinterpret_cast<char *>(&r.w));
    }
    VG_TRY(cudaMemcpy(out.blk_rec + total, pad2, sizeof(pad2), cudaMemcpyHostToDevice));
    VG_TRY(cudaGetLastError());
    VG_TRY(cudaDeviceSynchronize());
    out.blk_records = total + 2;
    out.seconds[1] = lap();
    // cell blocks
    int64_t *aoffs = nullptr, *foffs = nullptr;
    VG_TRY(tmp.get(&aoffs, M + 1));
    VG_TRY(tmp.get(&foffs, M + 1));
    cell_sizes_kernel<<<blocks_for(M, 256, in.sms), 256>>>(off, idx, M, aoffs, foffs);
    VG_TRY(launch_exclusive_scan(aoffs, M, scan, 0));
    VG_TRY(launch_exclusive_scan(foffs, M, scan, 0));
    int64_t na = 0, nf = 0;
    VG_TRY(cudaMemcpy(&na, aoffs + M, sizeof(int64_t), cudaMemcpyDeviceToHost));
    VG_TRY(cudaMemcpy(&nf, foffs + M, sizeof(int64_t), cudaMemcpyDeviceToHost));
    if (na + 8 >= ((int64_t)1 << 31) || nf + 8 >= ((int64_t)1 << 31)) {
        err = "cell blocks exceed 2^31 records";
        return LAYOUT_NOMEM;
    }
    VG_TRY(keep.get(&out.site, M));
    VG_TRY(keep.get(&out.cells, na + 8));
    VG_TRY(keep.get(&out.rel, nf + 8));
    out.ncells = na + 8;
    out.nrel = nf + 8;
    sites_kernel<<<blocks_for(M, 256, in.sms), 256>>>(s4, foffs, M, out.site);
    cell_blocks_kernel<<<blocks_for(M, kWarps, in.sms), wb>>>(s4, out.perm, off, idx, M, aoffs, foffs, in.unit, out.cells,
                                                             out.rel, reinterpret_cast<int *>(nbig + 1));
    tail_kernel<<<1, 8>>>(out.cells, na, out.rel, nf);
    // coarse density grid
    BlockDev dg = g;
    int64_t nd = 1;
    double vol = 1.0;
    for (int c = 0; c < 3; c++) {
        dg.dim[c] = in.ddim[c];
        nd *= in.ddim[c];
        vol *= ext[c];
    }
    unsigned *dcnt = nullptr;
    VG_TRY(tmp.get(&dcnt, nd));
    VG_TRY(keep.get(&out.dens, nd));
    VG_TRY(cudaMemset(dcnt, 0, sizeof(unsigned) * nd));
    density_count_kernel<<<blocks_for(M, 256, in.sms), 256>>>(s4, M, dg, dcnt);
    density_kernel<<<blocks_for(nd, 256, in.sms), 256>>>(dcnt, nd, vol / (double)nd, out.dens);
    count_launches(6);
    VG_TRY(cudaGetLastError());
    unsigned nb[3] = {0, 0, 0};
    VG_TRY(cudaMemcpy(nb, nbig, sizeof(nb), cudaMemcpyDeviceToHost));
    // the records of cells with very many neighbours: a handful, on the host
    if (nb[1]) {
        std::vector<int64_t> fo((size_t)M + 1);
        VG_TRY(cudaMemcpy(fo.data(), foffs, sizeof(int64_t) * (M + 1), cudaMemcpyDeviceToHost));
        for (int64_t i = 0; i < M; i++) {
            if (in.off[i + 1] - in.off[i] <= kMaxNeighbours) continue;
            int64_t n = 0;
            for (int64_t q = in.off[i]; q < in.off[i + 1]; q++) n += in.idx[q] >= 0;
            std::vector<float4> r((size_t)n);
            float4 *const list = out.rel + fo[i] + 2;
            VG_TRY(cudaMemcpy(r.data(), list, sizeof(float4) * n, cudaMemcpyDeviceToHost));
            std::sort(r.begin(), r.end(), [](const float4 &a, const float4 &b) {
                const double p = (double)a.x * a.x + (double)a.y * a.y + (double)a.z * a.z;
                const double q = (double)b.x * b.x + (double)b.y * b.y + (double)b.z * b.z;
                int32_t u, v;
                std::memcpy(&u, &a.w, 4);
                std::memcpy(&v, &b.w, 4);
                return p < q || (p == q && u < v);
            });
            VG_TRY(cudaMemcpy(list, r.data(), sizeof(float4) * n, cudaMemcpyHostToDevice));
        }
    }
    VG_TRY(cudaDeviceSynchronize());
    out.entries = total - nb[2];
    out.seconds[2] = lap();
    for (void *q : {(void *)out.site, (void *)out.cells, (void *)out.rel, (void *)out.perm, (void *)out.blk_off,
                    (void *)out.blk_rec, (void *)out.dens})
        keep.take(q);
    return LAYOUT_OK;
#undef VG_TRY
}

}  // namespace vg
