// GPU construction of the Voronoi cells: the parallel set-up the paper
// names as future work (Sect. 3.6). Same definition as the host builder: the
// cell of site m is the domain box cut by the bisector half-space of every
// site that can reach it (Sect. 2.1, Eq. 1-3); a site farther than twice the
// largest vertex radius cannot, so the search stops once every unvisited
// site is that far (security radius).
//
// Sites are first sorted into a grid of buckets (counting sort; each
// bucket's list is then ordered by site index so the result does not depend
// on atomic order). The grid lines of each axis sit at quantiles of the
// sites' coordinates on that axis, so that where the sites are dense the
// buckets are small: a density that is a product of functions of x, y and z
// gives every bucket about the same number of sites. One thread builds one cell: a convex polyhedron in
// float64 with shared vertices and faces as vertex loops, cut plane by plane
// while the buckets are visited ring by ring around the site, the sites of
// each ring nearest first. The polyhedron has fixed capacities; a cell that
// would overflow them is flagged and rebuilt by the host builder.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"
#include "kernels.h"

namespace vg {
namespace {

constexpr int kNV = 96;    // vertices of the polyhedron
constexpr int kNF = 48;    // faces
constexpr int kNL = 320;   // entries of all face loops
constexpr int kNE = 64;    // crossed edges of one cut
constexpr int kCap = 64;   // neighbour ids written back per cell

struct BucketGrid {
    const double *edge[3];  // grid lines of each axis: dim + 1 non-decreasing values, box bounds at both ends
    const float *line[3];   // the same in float32: exact but for the box bounds
    int dim[3];
};

struct Face {
    int id;
    short beg, len;
};

constexpr int kBuf = 384;  // candidates of one drain

// A thread's polyhedron and scratch: a run of global memory of its own. Local
// memory deals the threads' 4-byte words out in turn, so with the lanes of a warp
// at different cells (about 4 of 32 run together) every access moved a 32-byte
// sector for 4 bytes of it: 80 GB of DRAM traffic for 2 10^5 clumpy cells, 18 now,
// L1 hits 46 -> 81 %. Cell kernel 23.6 -> 15.8 ms at 10^5 clumpy sites, cell phase
// 138 -> 107 ms at 10^6. (32-byte vertices moved as pairs of double2: 2 % slower.)
struct Cell {
    struct {
        double x, y, z, f;  // f: the value of the cutting plane
    } v[kNV];
    Face face[kNF];
    unsigned char L[2][kNL];       // face loops: the current ones and those a cut writes
    unsigned long long key[kBuf];  // candidates: distance bits above the site
    float far[3 * kNV];            // the vertices a candidate can still cut
    unsigned char rank[kNV];       // order of the vertices
    // scratch of a cut
    int ekey[kNE];
    unsigned char evid[kNE];
    unsigned char seg_a[kNF], seg_b[kNF];
};
static_assert(sizeof(Cell) % 32 == 0, "every cell starts on a sector");

// the bucket of coordinate v along one axis: the largest i < dim with
// edge[i] <= v (0 below the first line)
template <class T>
__device__ __forceinline__ int bucket_coord(T v, const T *edge, int dim) {
    int lo = 0, hi = dim - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(edge + mid) <= v) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The grid lines of one axis: edge[i] is the (i n / dim)-th smallest of the n
// sampled coordinates (every stride-th site's; float32 values), the box bounds
// at both ends. One block per line finds the value whose rank it is, two bits at
// a time, each step counting the sample below three thresholds. Sorting the three
// samples on the host took 10 of the 37 ms of the cell phase at 10^5 sites.
// The counting is bound by the reads of the sample from L2, so it is laid out
// as one array of keys per axis (4 bytes a site instead of a strided float4),
// read 16 bytes a thread by 1024 threads; with one bit per step over the sites
// themselves and 256 threads it took 1006 us at 10^5 sites, 80 now.
constexpr int kLineThreads = 1024;

__device__ __forceinline__ unsigned float_order(float x) {  // orders like the value
    const unsigned b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : b | 0x80000000u;
}

// keys[c n4 + k]: coordinate c of sample k; n4 is n rounded up to a multiple of
// four, the rest of each array the largest key, which is below no threshold
__global__ void sample_keys_kernel(const float4 *Sf, int64_t stride, int n, int n4, unsigned *keys) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n4) return;
    unsigned x = 0xffffffffu, y = x, z = x;
    if (k < n) {
        const float4 q = __ldg(Sf + k * stride);
        x = float_order(q.x);
        y = float_order(q.y);
        z = float_order(q.z);
    }
    keys[k] = x;
    keys[n4 + k] = y;
    keys[2 * n4 + k] = z;
}

__global__ void __launch_bounds__(kLineThreads) grid_lines_kernel(const unsigned *keys, int n, int n4, int3 dims,
                                                                  double3 lo, double3 hi, double *edge, float *line) {
    __shared__ int s_count[3][kLineThreads / 32];
    const int dim[3] = {dims.x, dims.y, dims.z};
    int i = blockIdx.x, c = 0, first = 0;  // line i of axis c, dim + 1 lines each
    while (i > dim[c]) {
        i -= dim[c] + 1;
        first += dim[c] + 1;
        c++;
    }
    const double l = c == 0 ? lo.x : c == 1 ? lo.y : lo.z, h = c == 0 ? hi.x : c == 1 ? hi.y : hi.z;
    if (i == 0 || i == dim[c]) {
        if (threadIdx.x == 0) {
            edge[first + i] = i == 0 ? l : h;
            line[first + i] = (float)(i == 0 ? l : h);
        }
        return;
    }
    const int rank = (int)((int64_t)i * n / dim[c]);
    const uint4 *q4 = reinterpret_cast<const uint4 *>(keys + (int64_t)c * n4);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the largest key with at most `rank` keys below it
    unsigned key = 0u;
    for (int bit = 30; bit >= 0; bit -= 2) {
        const unsigned t1 = key | (1u << bit), t2 = key | (2u << bit), t3 = key | (3u << bit);
        int b1 = 0, b2 = 0, b3 = 0;
#pragma unroll 4
        for (int k = threadIdx.x; k < n4 / 4; k += kLineThreads) {
            const uint4 q = __ldg(q4 + k);
            b1 += (q.x < t1) + (q.y < t1) + (q.z < t1) + (q.w < t1);
            b2 += (q.x < t2) + (q.y < t2) + (q.z < t2) + (q.w < t2);
            b3 += (q.x < t3) + (q.y < t3) + (q.z < t3) + (q.w < t3);
        }
        b1 = __reduce_add_sync(0xffffffffu, b1);
        b2 = __reduce_add_sync(0xffffffffu, b2);
        b3 = __reduce_add_sync(0xffffffffu, b3);
        if (lane == 0) {
            s_count[0][warp] = b1;
            s_count[1][warp] = b2;
            s_count[2][warp] = b3;
        }
        __syncthreads();
        // every warp adds the warps' counts up for itself
        static_assert(kLineThreads == 1024, "one lane per warp's count");
        b1 = __reduce_add_sync(0xffffffffu, s_count[0][lane]);
        b2 = __reduce_add_sync(0xffffffffu, s_count[1][lane]);
        b3 = __reduce_add_sync(0xffffffffu, s_count[2][lane]);
        __syncthreads();
        key = b3 <= rank ? t3 : b2 <= rank ? t2 : b1 <= rank ? t1 : key;
    }
    if (threadIdx.x == 0) {
        const float v = __uint_as_float((key & 0x80000000u) ? key & 0x7fffffffu : ~key);
        edge[first + i] = fmin(fmax((double)v, l), h);
        line[first + i] = (float)edge[first + i];
    }
}

__global__ void bucket_count_kernel(const double *S, int64_t M, BucketGrid bg, int *bidx, int64_t *cnt) {
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M; m += (int64_t)gridDim.x * blockDim.x) {
        const int i = bucket_coord(S[3 * m], bg.edge[0], bg.dim[0]);
        const int j = bucket_coord(S[3 * m + 1], bg.edge[1], bg.dim[1]);
        const int k = bucket_coord(S[3 * m + 2], bg.edge[2], bg.dim[2]);
        const int b = (i * bg.dim[1] + j) * bg.dim[2] + k;
        bidx[m] = b;
        atomicAdd(reinterpret_cast<unsigned long long *>(&cnt[b]), 1ull);
    }
}

__global__ void bucket_fill_kernel(const int *bidx, int64_t M, int64_t *cursor, int *bsites) {
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M; m += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long at = atomicAdd(reinterpret_cast<unsigned long long *>(&cursor[bidx[m]]), 1ull);
        bsites[at] = (int)m;
    }
}

// order every bucket's list by site index (insertion sort; lists are short)
__global__ void bucket_sort_kernel(const int64_t *off, int64_t K, int *bsites) {
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < K; b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = off[b], e = off[b + 1];
        for (int64_t i = s + 1; i < e; i++) {
            const int v = bsites[i];
            int64_t k = i - 1;
            while (k >= s && bsites[k] > v) {
                bsites[k + 1] = bsites[k];
                k--;
            }
            bsites[k + 1] = v;
        }
    }
}

// The sites in bucket order, each with its index: the buckets of a row are one run
// of 16-byte entries, read four at a time. Before, each bucket's bounds, its
// sites' indices and their positions were three dependent reads one after the
// other, and every bucket of a ring was visited; rows and slabs of buckets out of
// reach are skipped now. The longest search binds a small grid: cell phase at
// 10^5 disk sites 32.4 -> 21.6 ms.
__global__ void bucket_sites_kernel(const float4 *Sf, const int *bsites, int64_t M, float4 *Sb) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < M; q += (int64_t)gridDim.x * blockDim.x) {
        const int m = bsites[q];
        const float4 p = __ldg(Sf + m);
        Sb[q] = make_float4(p.x, p.y, p.z, __int_as_float(m));
    }
}

// What a thread keeps of its polyhedron in registers. A vertex stays where it
// was made until a cut drops it, and new ones take the lowest free places; the
// order of the vertices, which decides the end that a new vertex is formed from,
// is a byte of its own, and the loops alternate between two arrays. Before, each
// cut renumbered the vertices, copied them to scratch and back and rewrote the
// loops: cell phase at 10^6 clumpy sites 103 -> 98 ms, 3 10^5 uniform ones 30.5 ->
// 28.7, at 10^5 the same within 1 %.
struct Counts {
    unsigned long long use0, use1;  // places taken
    int end;                        // places past the last one taken
    int nf, cur;                    // faces, and which loops are current
};
__device__ __forceinline__ bool bit128(unsigned long long m0, unsigned long long m1, int v) {
    return ((v < 64 ? m0 >> v : m1 >> (v - 64)) & 1ull) != 0ull;
}

__device__ void poly_box(Cell &P, Counts &C, const double *box) {
    C.use0 = 0xffull;
    C.use1 = 0ull;
    C.end = 8;
    for (int i = 0; i < 8; i++) {
        P.rank[i] = (unsigned char)i;
        P.v[i].x = (i & 4) ? box[3] : box[0];
        P.v[i].y = (i & 2) ? box[4] : box[1];
        P.v[i].z = (i & 1) ? box[5] : box[2];
    }
    // counter-clockwise seen from outside; walls -1..-6 = x min, x max, y min, y max, z min, z max
    const unsigned char quad[6][4] = {{0, 1, 3, 2}, {4, 6, 7, 5}, {0, 4, 5, 1}, {2, 3, 7, 6}, {0, 2, 6, 4}, {1, 5, 7, 3}};
    C.nf = 6;
    C.cur = 0;
    for (int w = 0; w < 6; w++) {
        P.face[w] = Face{-(w + 1), (short)(4 * w), 4};
        for (int k = 0; k < 4; k++) P.L[0][4 * w + k] = quad[w][k];
    }
}

// A double truncated to float32 with integer operations only (its high word:
// 21 significant bits, relative error below 2^-20; |x| < 2^-126 gives 0).
__device__ __forceinline__ float trunc_float(double x) {
    const int h = __double2hiint(x);
    const int e = (h >> 20) & 0x7ff;
    const int bits = (h & (int)0x80000000) | ((e - 896) << 23) | ((h & 0xfffff) << 3);
    return e > 896 ? __int_as_float(bits) : 0.0f;
}

// Cut P by {x : n.x <= d}. 1: changed, 0: untouched, -1: capacity exceeded
// or topology broken (the caller rebuilds the cell on the host).
__device__ int poly_cut(Cell &P, Counts &C, double nx, double ny, double nz, double d, int id, double eps) {
    // each vertex classified once: above the plane (fv > eps) and strictly
    // below it (fv < -eps) as bits of two 128-bit masks held in registers,
    // so that the face walk below tests the masks and reads fv only at the
    // two ends of an edge the plane cuts (eps > 0: compared as integers, off
    // the float64 pipe)
    static_assert(kNV <= 128, "vertex masks hold 128 bits");
    unsigned long long out0 = 0ull, out1 = 0ull, str0 = 0ull, str1 = 0ull;
    const long long eb = __double_as_longlong(eps);
    for (int i = 0; i < C.end; i++) {
        if (!bit128(C.use0, C.use1, i)) continue;
        const double f = nx * P.v[i].x + ny * P.v[i].y + nz * P.v[i].z - d;
        P.v[i].f = f;
        const long long fb = __double_as_longlong(f);
        const unsigned long long bit = 1ull << (i & 63);
        const unsigned long long ob = fb > eb ? bit : 0ull;
        const unsigned long long sb = fb < 0 && (fb & 0x7fffffffffffffffll) > eb ? bit : 0ull;
        if (i < 64) {
            out0 |= ob;
            str0 |= sb;
        } else {
            out1 |= ob;
            str1 |= sb;
        }
    }
    if (!(out0 | out1)) return 0;
    auto is_out = [&](int v) { return bit128(out0, out1, v); };
    auto is_strict = [&](int v) { return bit128(str0, str1, v); };
    const unsigned char *const L = P.L[C.cur];
    unsigned char *const L2 = P.L[C.cur ^ 1];
    unsigned long long free0 = ~C.use0, free1 = ~C.use1 & ((1ull << (kNV - 64)) - 1ull);
    int ne = 0, nseg = 0, nf2 = 0, nl2 = 0;
    for (int f = 0; f < C.nf; f++) {
        const Face fc = P.face[f];
        const int b = fc.beg, k = fc.len;
        const int start = nl2;
        int entry = -1, exit_ = -1;
        // one pass: a face wholly above the plane leaves no entries
        int vb = L[b];
        bool bo = is_out(vb);
        for (int i = 1; i <= k; i++) {
            const int va = vb;
            const bool ao = bo;
            vb = L[b + (i < k ? i : 0)];
            bo = is_out(vb);
            if (!ao) {
                if (nl2 >= kNL) return -1;
                L2[nl2++] = (unsigned char)va;
            }
            if (ao != bo) {
                const bool strict = !ao ? is_strict(va) : is_strict(vb);
                int x = !ao ? va : vb;
                if (strict) {
                    // the vertex on edge (va, vb), made once from the lower index
                    const bool up = P.rank[va] < P.rank[vb];
                    const int lo = up ? va : vb, hi = up ? vb : va;
                    const int key = lo * 256 + hi;
                    x = -1;
                    for (int e = 0; e < ne; e++)
                        if (P.ekey[e] == key) { x = P.evid[e]; break; }
                    if (x < 0) {
                        if (ne >= kNE || !(free0 | free1)) return -1;
                        x = free0 ? __ffsll((long long)free0) - 1 : 63 + __ffsll((long long)free1);
                        if (free0) free0 &= free0 - 1;
                        else free1 &= free1 - 1;
                        const auto vl = P.v[lo], vh = P.v[hi];
                        const double t = vl.f / (vl.f - vh.f);
                        P.v[x].x = vl.x + t * (vh.x - vl.x);
                        P.v[x].y = vl.y + t * (vh.y - vl.y);
                        P.v[x].z = vl.z + t * (vh.z - vl.z);
                        P.ekey[ne] = key;
                        P.evid[ne] = (unsigned char)x;
                        ne++;
                    }
                    if (nl2 >= kNL) return -1;
                    L2[nl2++] = (unsigned char)x;
                }
                if (!ao) exit_ = x;
                else entry = x;
            }
        }
        if (entry >= 0 && exit_ >= 0 && entry != exit_) {
            if (nseg >= kNF) return -1;
            P.seg_a[nseg] = (unsigned char)entry;
            P.seg_b[nseg] = (unsigned char)exit_;
            nseg++;
        }
        if (nl2 > start && nf2 >= kNF) return -1;
        if (nl2 - start >= 3) {
            P.face[nf2++] = Face{fc.id, (short)start, (short)(nl2 - start)};
        } else {
            nl2 = start;
        }
    }
    if (nseg > 0) {
        // cap face: chain the cut segments entry -> exit
        const int start = nl2;
        int cur = P.seg_a[0];
        const int first = cur;
        bool ok = true;
        unsigned long long used = 0ull;
        for (int step = 0; step < nseg; step++) {
            int pick = -1;
            for (int i = 0; i < nseg; i++)
                if (!((used >> i) & 1ull) && P.seg_a[i] == cur) { pick = i; break; }
            if (pick < 0) { ok = false; break; }
            used |= 1ull << pick;
            if (nl2 >= kNL) return -1;
            L2[nl2++] = P.seg_a[pick];
            cur = P.seg_b[pick];
        }
        if (!ok || cur != first) return -1;  // inconsistent topology: leave it to the host
        if (nl2 - start >= 3) {
            if (nf2 >= kNF) return -1;
            P.face[nf2++] = Face{id, (short)start, (short)(nl2 - start)};
        } else {
            nl2 = start;
        }
    }
    // the vertices still referenced, ranked by their first place in the loops
    unsigned long long met0 = 0ull, met1 = 0ull;
    int n = 0;
    for (int i = 0; i < nl2; i++) {
        const int v = L2[i];
        if (bit128(met0, met1, v)) continue;
        if (v < 64) met0 |= 1ull << v;
        else met1 |= 1ull << (v - 64);
        P.rank[v] = (unsigned char)n++;
    }
    C.use0 = met0;
    C.use1 = met1;
    C.end = met1 ? 128 - __clzll((long long)met1) : 64 - __clzll((long long)met0);
    C.cur ^= 1;
    C.nf = nf2;
    return nf2 >= 4 ? 1 : -1;
}

// Persistent threads: each takes its next cell from a global counter as soon
// as it has finished one, so a thread whose cell needed few cuts does not
// wait for the slowest cell of its block. Eight blocks of 128 per SM (64
// registers): the kernel waits on its polyhedra and gains more from the extra
// warps than it loses to the spills where cells are many (cell phase at 10^6
// clumpy sites: 98 ms, 101 with six blocks, 106 with five; 10^5 clumpy: 20.8, 18.7
// and 18.5, but 10^5 disk sites 21.7, 22.9 and 22.5 and 10^4 clumpy 4.82, 5.01 and
// 5.03).
__global__ void __launch_bounds__(128, 8) cells_kernel(const double *S, int64_t M, BucketGrid bg, const int64_t *boff,
                                                    const float4 *Sb, double box0, double box1, double box2,
                                                    double box3, double box4, double box5, double eps, int *out_cnt,
                                                    int *out_nbr, double *out_vol, double *out_bbox, int *out_fail,
                                                    unsigned long long *next, const float4 *Sf, int lanes,
                                                    Cell *pool) {
    if ((int)(threadIdx.x & 31) >= lanes) return;  // few cells: fewer lanes in more warps (see the launch)
    Cell &P = pool[(int64_t)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * lanes + (threadIdx.x & 31)];
    Counts C;
    const double box[6] = {box0, box1, box2, box3, box4, box5};
    double X = 0.0;
    for (int c = 0; c < 6; c++) X = fmax(X, fabs(box[c]));
    const float Xf = __double2float_ru(X);
    const float off = Xf * 0x1p-19f;  // a truncated vertex is off by less (three components of 2^-20 X)
    for (int64_t m = (int64_t)atomicAdd(next, 1ull); m < M; m = (int64_t)atomicAdd(next, 1ull)) {
        const double px = S[3 * m], py = S[3 * m + 1], pz = S[3 * m + 2];
        poly_box(P, C, box);
        // Float32 work that keeps most candidates off the float64 pipe, which a
        // warp pays for all its lanes whenever one of them uses it. Sites are
        // float32 values, so pf and the candidates are exact.
        //  * reach: a site farther than twice the largest vertex radius cannot
        //    cut the cell. The radius comes from the truncated vertices, rounded
        //    up; squared distances are within 2^-21 of the exact ones, and a site
        //    is dropped only beyond reach^2 (1 + 2^-17).
        //  * far vertices: a candidate at distance D can only cut vertices at
        //    least D/2 from the site, so with candidates taken nearest first a
        //    shrinking list of vertices (P.far) has to be tested.
        //  * screen: the candidate's plane n.v = n.p + |n|^2/2 (n not normalised)
        //    against those vertices. Truncation and rounding leave n.v and the
        //    right side within |n|_1 X 2^-19; a candidate is dropped when every
        //    vertex lies below by |n|_1 X 2^-18, where the float64 test finds no
        //    vertex above the plane either.
        // Before, every candidate within reach was normalised (a square root and
        // three divisions in float64) ahead of a screen over all vertices, and
        // the largest radius taken in float64 after each cut: 30,000 sites in a
        // ball, whose surface cells reach the corners of the box and meet tens of
        // thousands of candidates, took 409 ms instead of 137, 10^5 disk sites 55
        // instead of 52, 10^6 clumpy ones 159 instead of 144 (cell phase, with the
        // polyhedra still in local memory; the last two take 21 and 97 ms now).
        const float4 pf = Sf[m];
        float R2f = 0.f, reach = 0.f;
        int nfar = 0;
        auto refresh = [&](float d2min) {
            const float hm = fmaxf(0.5f * (1.0f - 0x1p-18f) * __fsqrt_rd(d2min) - off, 0.0f);
            const float hm2 = __fmul_rd(hm, hm);
            float r2 = 0.f;
            nfar = 0;
            for (int i = 0; i < C.end; i++) {
                if (!bit128(C.use0, C.use1, i)) continue;
                const float vx = trunc_float(P.v[i].x), vy = trunc_float(P.v[i].y), vz = trunc_float(P.v[i].z);
                const float dx = vx - pf.x, dy = vy - pf.y, dz = vz - pf.z;
                const float r = __fmaf_ru(dz, dz, __fmaf_ru(dy, dy, __fmul_ru(dx, dx)));
                r2 = fmaxf(r2, r);
                if (r >= hm2) {
                    P.far[3 * nfar] = vx;
                    P.far[3 * nfar + 1] = vy;
                    P.far[3 * nfar + 2] = vz;
                    nfar++;
                }
            }
            reach = __fmaf_ru(2.0f, __fadd_ru(__fsqrt_ru(r2), off), 4.0f * (float)eps);
            R2f = __fmul_ru(__fmul_ru(reach, reach), 1.0f + 0x1p-17f);
        };
        refresh(0.0f);
        const int bi = bucket_coord(pf.x, bg.line[0], bg.dim[0]);
        const int bj = bucket_coord(pf.y, bg.line[1], bg.dim[1]);
        const int bk = bucket_coord(pf.z, bg.line[2], bg.dim[2]);
        const int smax = max(bg.dim[0], max(bg.dim[1], bg.dim[2]));
        int fail = 0;
        // each shell's candidates within reach are cut nearest first (up to
        // kBuf at a time, picked by float32 distance, ties by index): the
        // near planes shrink the polyhedron, and with it the reach, so that
        // more of the far candidates drop out before they are cut. The
        // result is the same polyhedron up to rounding; only the work to
        // reach it changes. A candidate is one 64-bit key, the distance's
        // bits above the site index (non-negative floats order as their
        // bits), and the buffer becomes a binary min-heap when it is
        // drained, so each pick costs a walk down the heap rather than a
        // scan of the whole buffer.
        int nb = 0;
        auto sift_down = [&](int i, unsigned long long v) {
            for (;;) {
                int c = 2 * i + 1;
                if (c >= nb) break;
                unsigned long long cv = P.key[c];
                if (c + 1 < nb) {
                    const unsigned long long c2 = P.key[c + 1];
                    if (c2 < cv) { cv = c2; c++; }
                }
                if (v <= cv) break;
                P.key[i] = cv;
                i = c;
            }
            P.key[i] = v;
        };
        auto flush = [&]() -> int {
            if (nb == 0) return 0;
            for (int i = nb / 2 - 1; i >= 0; i--) sift_down(i, P.key[i]);
            refresh(__uint_as_float((unsigned)(P.key[0] >> 32)));
            while (nb > 0) {
                const unsigned long long top = P.key[0];
                nb--;
                if (nb > 0) sift_down(0, P.key[nb]);
                const float d2k = __uint_as_float((unsigned)(top >> 32));
                const int jj = (int)(unsigned)top;
                if (d2k > R2f) {
                    nb = 0;  // the nearest left is out of reach: so are the others
                    break;
                }
                {
                    const float4 qf = Sf[jj];
                    const float fx = qf.x - pf.x, fy = qf.y - pf.y, fz = qf.z - pf.z;
                    const float n1 = fabsf(fx) + fabsf(fy) + fabsf(fz);
                    const float np = __fmaf_rn(fz, pf.z, __fmaf_rn(fy, pf.y, __fmul_rn(fx, pf.x)));
                    const float T = __fadd_rn(np, __fmaf_rn(0.5f, d2k, -n1 * Xf * 0x1p-18f));
                    bool maybe = false;
                    for (int i = 0; i < nfar && !maybe; i++) {
                        const float v = __fmaf_rn(fz, P.far[3 * i + 2],
                                                  __fmaf_rn(fy, P.far[3 * i + 1], __fmul_rn(fx, P.far[3 * i])));
                        maybe = !(v <= T);
                    }
                    if (!maybe) continue;
                }
                const double qx = S[3 * (int64_t)jj], qy = S[3 * (int64_t)jj + 1], qz = S[3 * (int64_t)jj + 2];
                const double dx = qx - px, dy = qy - py, dz = qz - pz;
                const double dist = sqrt(dx * dx + dy * dy + dz * dz);
                const double nx = dx / dist, ny = dy / dist, nz = dz / dist;
                const double d = nx * 0.5 * (qx + px) + ny * 0.5 * (qy + py) + nz * 0.5 * (qz + pz);
                const int rc = poly_cut(P, C, nx, ny, nz, d, jj, eps);
                if (rc < 0) return 1;
                if (rc > 0) refresh(d2k);
            }
            return 0;
        };
        // one run of the sites in bucket order: those within reach go into the buffer
        auto scan = [&](int64_t q, int64_t end) -> int {
            for (; q < end; q += 4) {
                float4 c[4];
#pragma unroll
                for (int u = 0; u < 4; u++) c[u] = __ldg(Sb + min(q + u, end - 1));
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    const float fx = __fsub_rn(c[u].x, pf.x), fy = __fsub_rn(c[u].y, pf.y), fz = __fsub_rn(c[u].z, pf.z);
                    const float d2f = __fmaf_rn(fz, fz, __fmaf_rn(fy, fy, __fmul_rn(fx, fx)));
                    const int jj = __float_as_int(c[u].w);
                    if (q + u >= end || d2f > R2f || jj == (int)m) continue;
                    if (nb == kBuf && flush()) return 1;
                    P.key[nb++] = ((unsigned long long)__float_as_uint(d2f) << 32) | (unsigned)jj;
                }
            }
            return 0;
        };
        // Distance along one axis from the site to the sites of bucket i (edge[i] <= v
        // <= edge[i + 1]), rounded down. A slab or row of buckets is skipped where it
        // takes every site beyond reach by more than the rounding of d2f (2^-21).
        // In float32, as the ring's gap below: the lines are float32 values, and the
        // float64 pipe is the kernel's second limit (10^5 disk sites 21.6 -> 20.8 ms,
        // 10^5 clumpy 20.4 -> 20.1).
        auto off_axis = [&](int c, int i) {
            const float p = c == 0 ? pf.x : pf.y;
            const float *e = bg.line[c] + i;
            return fmaxf(fmaxf(__fsub_rd(__ldg(e), p), __fsub_rd(p, __ldg(e + 1))), 0.0f);
        };
        for (int s = 0; s <= smax && !fail; s++) {
            for (int i = max(bi - s, 0); i <= min(bi + s, bg.dim[0] - 1) && !fail; i++) {
                const float ox = off_axis(0, i), ox2 = __fmul_rd(ox, ox);
                if (ox2 * (1.0f - 0x1p-19f) > R2f) continue;
                for (int j = max(bj - s, 0); j <= min(bj + s, bg.dim[1] - 1) && !fail; j++) {
                    const float oy = off_axis(1, j);
                    if (__fmaf_rd(oy, oy, ox2) * (1.0f - 0x1p-19f) > R2f) continue;
                    const int64_t *row = boff + (int64_t)(i * bg.dim[1] + j) * bg.dim[2];
                    // a row of the shell is one run; inside the shell its two ends are
                    const bool shell = abs(i - bi) == s || abs(j - bj) == s;
                    for (int r = 0; r < (shell ? 1 : 2) && !fail; r++) {
                        int k0 = r == 0 ? bk - s : bk + s, k1 = shell ? bk + s : k0;
                        if (shell) {
                            k0 = max(k0, 0);
                            k1 = min(k1, bg.dim[2] - 1);
                        } else if (k0 < 0 || k0 >= bg.dim[2]) {
                            continue;
                        }
                        fail = scan(__ldg(row + k0), __ldg(row + k1 + 1));
                    }
                }
            }
            if (!fail) fail = flush();
            // every unvisited site lies beyond one of the grid lines that
            // bound rings 0..s (a site in bucket i has edge[i] <= v <
            // edge[i + 1]), so it is at least the smallest gap from the
            // site to those lines away; there are no sites past the last
            // bucket on either side
            float gap = INFINITY;
            for (int c = 0; c < 3; c++) {
                const float p = c == 0 ? pf.x : c == 1 ? pf.y : pf.z;
                const int b = c == 0 ? bi : c == 1 ? bj : bk;
                if (b + s + 1 <= bg.dim[c] - 1) gap = fminf(gap, __fsub_rd(__ldg(bg.line[c] + b + s + 1), p));
                if (b - s >= 1) gap = fminf(gap, __fsub_rd(p, __ldg(bg.line[c] + b - s)));
            }
            if (reach < gap) break;
        }
        // faces of positive area -> neighbours; volume as pyramids from the site; bounding box
        static_assert(kNE >= kCap, "the edge keys hold the neighbour list");
        int *const ids = P.ekey;  // free once the cuts are done
        int cnt = 0;
        double vol = 0.0;
        double bb[6] = {1e300, 1e300, 1e300, -1e300, -1e300, -1e300};
        const unsigned char *const L = P.L[C.cur];
        for (int f = 0; f < C.nf && !fail; f++) {
            const Face fc = P.face[f];
            const int b = fc.beg, k = fc.len;
            const int v0 = L[b];
            double sx = 0, sy = 0, sz = 0, sv = 0;
            for (int t = 1; t + 1 < k; t++) {
                const int v1 = L[b + t], v2 = L[b + t + 1];
                const double ax = P.v[v1].x - P.v[v0].x, ay = P.v[v1].y - P.v[v0].y, az = P.v[v1].z - P.v[v0].z;
                const double cx = P.v[v2].x - P.v[v0].x, cy = P.v[v2].y - P.v[v0].y, cz = P.v[v2].z - P.v[v0].z;
                const double ux = ay * cz - az * cy, uy = az * cx - ax * cz, uz = ax * cy - ay * cx;
                sx += ux;
                sy += uy;
                sz += uz;
                // signed volume of the tetrahedron (site, v0, v1, v2)
                sv += ((P.v[v0].x - px) * ux + (P.v[v0].y - py) * uy + (P.v[v0].z - pz) * uz) / 6.0;
            }
            vol += fabs(sv);
            const double area2 = sx * sx + sy * sy + sz * sz;
            if (area2 > 0.0) {
                if (cnt >= kCap) { fail = 1; break; }
                ids[cnt++] = fc.id;
            }
        }
        for (int i = 0; i < C.end; i++) {
            if (!bit128(C.use0, C.use1, i)) continue;
            bb[0] = fmin(bb[0], P.v[i].x);
            bb[1] = fmin(bb[1], P.v[i].y);
            bb[2] = fmin(bb[2], P.v[i].z);
            bb[3] = fmax(bb[3], P.v[i].x);
            bb[4] = fmax(bb[4], P.v[i].y);
            bb[5] = fmax(bb[5], P.v[i].z);
        }
        // the list in ascending order without repeats (insertion sort: a few
        // dozen ids), as the host's CSR holds it
        for (int a = 1; a < cnt; a++) {
            const int v = ids[a];
            int b = a - 1;
            while (b >= 0 && ids[b] > v) {
                ids[b + 1] = ids[b];
                b--;
            }
            ids[b + 1] = v;
        }
        int u = 0;
        for (int a = 0; a < cnt; a++)
            if (u == 0 || ids[a] != ids[u - 1]) ids[u++] = ids[a];
        for (int a = 0; a < u; a++) out_nbr[m * kCap + a] = ids[a];
        out_cnt[m] = u;
        out_vol[m] = vol;
        for (int c = 0; c < 6; c++) out_bbox[6 * m + c] = bb[c];
        out_fail[m] = fail;
    }
}

// the cells' lists into one CSR array (offsets computed on the host)
__global__ void gather_lists_kernel(const int *nbr, const int *cnt, const int64_t *off, int64_t M, int *idx) {
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M; m += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = off[m];
        const int c = cnt[m];
        for (int a = 0; a < c; a++) idx[o + a] = nbr[m * kCap + a];
    }
}

}  // namespace

int build_cells_gpu(const double *S, int64_t M, const double *box, int threads, CellsOut &out, std::string &err,
                    int64_t *host_fallback_cells) {
    // the float32 filters square and multiply coordinates: outside the range
    // where that is safe the problem is scaled by a power of two (exact), and
    // the volumes and bounding boxes are scaled back
    {
        double X = 0.0;
        for (int c = 0; c < 6; c++) X = std::max(X, std::fabs(box[c]));
        if (X < 0x1p-30 || X > 0x1p30) {
            const int k = -std::ilogb(X);
            std::vector<double> T(3 * (size_t)M);
            for (int64_t i = 0; i < 3 * M; i++) T[i] = std::ldexp(S[i], k);
            double tb[6];
            for (int c = 0; c < 6; c++) tb[c] = std::ldexp(box[c], k);
            const int rc = build_cells_gpu(T.data(), M, tb, threads, out, err, host_fallback_cells);
            if (out.d_bbox) cudaFree(out.d_bbox);
            out.d_bbox = nullptr;  // scaled
            for (double &v : out.vol) v = std::ldexp(v, -3 * k);
            for (double &v : out.bbox) v = std::ldexp(v, -k);
            return rc;
        }
    }
    const double ext[3] = {box[3] - box[0], box[4] - box[1], box[5] - box[2]};
    const double diag = std::sqrt(ext[0] * ext[0] + ext[1] * ext[1] + ext[2] * ext[2]);
    const double eps = 1e-12 * diag;
    BucketGrid bg;
    const double target = std::max(1.0, 0.5 * (double)M);  // about two sites per bucket
    const double w = std::cbrt(ext[0] * ext[1] * ext[2] / target);
    int64_t K = 1;
    // grid lines at quantiles of each coordinate, from every stride-th site
    // (fewer than 2^17 of them; deterministic)
    const int64_t stride = std::max<int64_t>(1, M >> 16);
    int64_t lines = 0;
    for (int c = 0; c < 3; c++) {
        bg.dim[c] = (int)std::min<long>(std::max<long>(std::lround(ext[c] / w), 1), 512);
        K *= bg.dim[c];
        lines += bg.dim[c] + 1;
    }
    double *dS = nullptr, *dE = nullptr;
    float4 *dSf = nullptr, *dSb = nullptr;
    int *bidx = nullptr, *bsites = nullptr, *cnt = nullptr, *nbr = nullptr, *fail = nullptr;
    int64_t *boff = nullptr, *cursor = nullptr, *tmp = nullptr, *doff = nullptr;
    int *didx = nullptr;
    Cell *pool = nullptr;
    double *vol = nullptr, *bbox = nullptr;
    auto cleanup = [&]() {
        void *ptrs[] = {dS, dE, dSf, dSb, bidx, bsites, cnt, nbr, fail, boff, cursor, tmp, vol, bbox, doff, didx, pool};
        for (void *p : ptrs)
            if (p) cudaFree(p);
    };
    auto bad = [&](cudaError_t e, const char *what) {
        err = std::string("GPU cell construction: ") + what + ": " + cudaGetErrorString(e);
        cudaGetLastError();  // or the next launch's check would report it
        cleanup();
        return -1;
    };
    cudaError_t e;
    if ((e = cudaMalloc(&dS, sizeof(double) * 3 * M)) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&bidx, sizeof(int) * M)) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&bsites, sizeof(int) * M)) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&boff, sizeof(int64_t) * (K + 1))) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&cursor, sizeof(int64_t) * (K + 1))) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&tmp, sizeof(int64_t) * scan_tmp_elems(K))) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&cnt, sizeof(int) * M)) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&nbr, sizeof(int) * kCap * M)) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&fail, sizeof(int) * M)) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&vol, sizeof(double) * M)) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMalloc(&bbox, sizeof(double) * 6 * M)) != cudaSuccess) return bad(e, "alloc");
    if ((e = cudaMemcpy(dS, S, sizeof(double) * 3 * M, cudaMemcpyHostToDevice)) != cudaSuccess) return bad(e, "upload");
    if ((e = cudaMalloc(&dE, (sizeof(double) + sizeof(float)) * lines)) != cudaSuccess) return bad(e, "alloc");
    bg.edge[0] = dE;
    bg.edge[1] = dE + bg.dim[0] + 1;
    bg.edge[2] = bg.edge[1] + bg.dim[1] + 1;
    float *const dl = reinterpret_cast<float *>(dE + lines);
    for (int c = 0; c < 3; c++) bg.line[c] = dl + (bg.edge[c] - dE);
    {
        // float copies of the sites (float32 values, or scaled ones: exact)
        std::vector<float4> sf((size_t)M);
        for (int64_t m = 0; m < M; m++)
            sf[m] = make_float4((float)S[3 * m], (float)S[3 * m + 1], (float)S[3 * m + 2], 0.f);
        if ((e = cudaMalloc(&dSf, sizeof(float4) * M)) != cudaSuccess) return bad(e, "alloc");
        if ((e = cudaMalloc(&dSb, sizeof(float4) * M)) != cudaSuccess) return bad(e, "alloc");
        if ((e = cudaMemcpy(dSf, sf.data(), sizeof(float4) * M, cudaMemcpyHostToDevice)) != cudaSuccess)
            return bad(e, "upload");
    }
    {
        // the keys lie in the lists' buffer (64 M ints), which the cells fill later
        static_assert(kCap >= 12, "3 (n + 3) keys, n <= M");
        const int n = (int)((M + stride - 1) / stride), n4 = (n + 3) & ~3;
        unsigned *const keys = reinterpret_cast<unsigned *>(nbr);
        sample_keys_kernel<<<(unsigned)((n4 + 255) / 256), 256>>>(dSf, stride, n, n4, keys);
        grid_lines_kernel<<<(unsigned)lines, kLineThreads>>>(keys, n, n4, make_int3(bg.dim[0], bg.dim[1], bg.dim[2]),
                                                             make_double3(box[0], box[1], box[2]),
                                                             make_double3(box[3], box[4], box[5]), dE, dl);
    }
    if ((e = cudaMemset(boff, 0, sizeof(int64_t) * (K + 1))) != cudaSuccess) return bad(e, "memset");
    const int blocks = (int)std::min<int64_t>((M + 255) / 256, 65535);
    bucket_count_kernel<<<blocks, 256>>>(dS, M, bg, bidx, boff);
    if ((e = launch_exclusive_scan(boff, K, tmp, 0)) != cudaSuccess) return bad(e, "scan");
    if ((e = cudaMemcpy(cursor, boff, sizeof(int64_t) * (K + 1), cudaMemcpyDeviceToDevice)) != cudaSuccess)
        return bad(e, "copy");
    bucket_fill_kernel<<<blocks, 256>>>(bidx, M, cursor, bsites);
    bucket_sort_kernel<<<(int)std::min<int64_t>((K + 255) / 256, 65535), 256>>>(boff, K, bsites);
    bucket_sites_kernel<<<blocks, 256>>>(dSf, bsites, M, dSb);
    int dev = 0, sms = 1, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cells_kernel, 128, 0) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    // The lanes of a warp take turns wherever their cells differ, so few cells
    // are spread over all warps that fit, down to one cell per warp: 1000 cells
    // take 2.3 ms instead of 6.1, 10^4 clumpy ones 8.2 instead of 14.6 (cell phase,
    // with the polyhedra still in local memory; 10^4 take 4.7 now).
    const int lanes = (int)std::min<int64_t>(32, std::max<int64_t>(1, M / ((int64_t)sms * 32)));
    const int64_t per_block = 4 * lanes;
    int cblocks = (int)std::max<int64_t>(1, std::min<int64_t>((M + per_block - 1) / per_block, (int64_t)per_sm * sms));
    if ((e = cudaMemset(cursor, 0, sizeof(unsigned long long))) != cudaSuccess) return bad(e, "memset");
    // 1.4 GB for a GPU full of threads; with less room, fewer threads take turns
    while ((e = cudaMalloc(&pool, sizeof(Cell) * cblocks * per_block)) != cudaSuccess) {
        if (cblocks == 1) return bad(e, "alloc");
        cudaGetLastError();
        cblocks /= 2;
    }
    cells_kernel<<<cblocks, 128>>>(dS, M, bg, boff, dSb, box[0], box[1], box[2], box[3], box[4], box[5], eps, cnt,
                                   nbr, vol, bbox, fail, reinterpret_cast<unsigned long long *>(cursor), dSf, lanes, pool);
    count_launches(7);  // keys, grid lines, bucket count, fill, sort, sites, cells (the scan counts its own)
    if ((e = cudaDeviceSynchronize()) != cudaSuccess) return bad(e, "cells kernel");
    std::vector<int> hcnt(M), hfail(M);
    out.vol.assign(M, 0.0);
    out.bbox.assign(6 * M, 0.0);
    if ((e = cudaMemcpy(hcnt.data(), cnt, sizeof(int) * M, cudaMemcpyDeviceToHost)) != cudaSuccess ||
        (e = cudaMemcpy(hfail.data(), fail, sizeof(int) * M, cudaMemcpyDeviceToHost)) != cudaSuccess ||
        (e = cudaMemcpy(out.vol.data(), vol, sizeof(double) * M, cudaMemcpyDeviceToHost)) != cudaSuccess ||
        (e = cudaMemcpy(out.bbox.data(), bbox, sizeof(double) * 6 * M, cudaMemcpyDeviceToHost)) != cudaSuccess)
        return bad(e, "download");
    if (std::find(hfail.begin(), hfail.end(), 1) == hfail.end()) {
        // every cell was built here: its list is sorted already, so only the
        // CSR is gathered on the device and read back
        out.off.assign(M + 1, 0);
        for (int64_t m = 0; m < M; m++) out.off[m + 1] = out.off[m] + hcnt[m];
        out.idx.resize(out.off[M]);
        if (host_fallback_cells) *host_fallback_cells = 0;
        if ((e = cudaMalloc(&doff, sizeof(int64_t) * (M + 1))) != cudaSuccess) return bad(e, "alloc");
        if ((e = cudaMalloc(&didx, sizeof(int) * std::max<int64_t>(1, out.off[M]))) != cudaSuccess)
            return bad(e, "alloc");
        if ((e = cudaMemcpy(doff, out.off.data(), sizeof(int64_t) * (M + 1), cudaMemcpyHostToDevice)) != cudaSuccess)
            return bad(e, "upload");
        gather_lists_kernel<<<blocks, 256>>>(nbr, cnt, doff, M, didx);
        count_launches(1);
        if ((e = cudaMemcpy(out.idx.data(), didx, sizeof(int) * out.off[M], cudaMemcpyDeviceToHost)) != cudaSuccess)
            return bad(e, "download");
        out.d_off = doff;
        out.d_idx = didx;
        out.d_bbox = bbox;
        doff = nullptr;
        didx = nullptr;
        bbox = nullptr;
        cleanup();
        return 0;
    }
    std::vector<int> hnbr((size_t)kCap * M);
    if ((e = cudaMemcpy(hnbr.data(), nbr, sizeof(int) * kCap * M, cudaMemcpyDeviceToHost)) != cudaSuccess)
        return bad(e, "download");
    cleanup();
    // each cell's list sorted and made unique in place (parallel over
    // cells), the failed cells rebuilt on the host, then one CSR
    std::vector<int64_t> len(M, 0);
    parallel_for(M, threads, 1 << 12, [&](int64_t b, int64_t e) {
        for (int64_t m = b; m < e; m++) {
            if (hfail[m]) continue;
            int *row = hnbr.data() + m * kCap;
            std::sort(row, row + hcnt[m]);
            len[m] = std::unique(row, row + hcnt[m]) - row;
        }
    });
    std::vector<int32_t> redo;
    for (int64_t m = 0; m < M; m++)
        if (hfail[m]) redo.push_back((int32_t)m);
    if (host_fallback_cells) *host_fallback_cells = (int64_t)redo.size();
    std::vector<std::vector<int32_t>> lists(redo.empty() ? 0 : M);
    if (!redo.empty()) {
        if (build_cells_into(S, M, box, threads, &redo, lists, out.vol.data(), out.bbox.data(), err) != 0) return -1;
        for (int32_t m : redo) len[m] = (int64_t)lists[m].size();
    }
    out.off.assign(M + 1, 0);
    for (int64_t m = 0; m < M; m++) out.off[m + 1] = out.off[m] + len[m];
    out.idx.resize(out.off[M]);
    parallel_for(M, threads, 1 << 12, [&](int64_t b, int64_t e) {
        for (int64_t m = b; m < e; m++) {
            if (hfail[m]) std::copy(lists[m].begin(), lists[m].end(), out.idx.begin() + out.off[m]);
            else std::copy(hnbr.begin() + m * kCap, hnbr.begin() + m * kCap + len[m], out.idx.begin() + out.off[m]);
        }
    });
    return 0;
}

}  // namespace vg
