// Evaluation of a fit (Sec. 4): the zero level set of a grid field as
// triangles, area-weighted samples on it, and the point-to-point surface
// metrics HD, CD and CS between two sampled surfaces; plus the inverse of
// Eq. 3-10 and an index scatter to bring binned results back to grid order.
//
// The paper extracts the surface with marching cubes; here every grid cube
// is split into six tetrahedra {0, a, a + b, 7} (corner bits x = 1, y = 2,
// z = 4; axis orders (a, b) = (1,2) (1,4) (2,1) (2,4) (4,1) (4,2)), which needs
// no case table.  Inside means value < iso.  A tetrahedron with one or three
// inside vertices gives one triangle on the lone vertex's three edges, with
// two it gives the quad on the four crossing edges as two triangles.  Edge
// points interpolate from the edge's lower grid index to the higher one in
// float with a fixed operation order, so results are reproducible bit for
// bit and a shared edge gives the same point everywhere.  Output is in cube
// order (counts, exclusive scan, write).
#include <math.h>

#include "common.cuh"

using namespace serbf;

namespace {

__constant__ int c_tets[6][4] = {{0, 1, 3, 7}, {0, 1, 5, 7}, {0, 2, 3, 7}, {0, 2, 6, 7}, {0, 4, 5, 7}, {0, 4, 6, 7}};

struct Grid3 {
    int nx, ny, nz;
    float o[3];
    float h;
};

// A cube's lower corner and its eight values (corner c: bits x, y, z).
struct Cube {
    int i, j, k;
    float f[8];
};

__device__ __forceinline__ Cube cube_at(const float *f, const Grid3 &g, int64_t c) {
    Cube q;
    const int cx = g.nx - 1, cy = g.ny - 1;
    const int64_t row = c / cx;
    q.i = (int)(c - row * cx);
    q.k = (int)(row / cy);
    q.j = (int)(row - (int64_t)q.k * cy);
    const float *p = f + ((int64_t)q.k * g.ny + q.j) * g.nx + q.i;
    const int64_t up = (int64_t)g.ny * g.nx;
#pragma unroll
    for (int b = 0; b < 8; ++b) q.f[b] = p[(b & 1) + ((b >> 1) & 1) * g.nx + (b >> 2) * up];
    return q;
}

// Corners below iso, one bit each.
__device__ __forceinline__ int inside(const Cube &q, float iso) {
    int m = 0;
#pragma unroll
    for (int b = 0; b < 8; ++b) m |= (q.f[b] < iso) << b;
    return m;
}

__device__ __forceinline__ int tet_mask(int in, int t) {
    return ((in >> c_tets[t][0]) & 1) | ((in >> c_tets[t][1]) & 1) << 1 | ((in >> c_tets[t][2]) & 1) << 2 |
           ((in >> c_tets[t][3]) & 1) << 3;
}

__device__ __forceinline__ int tris_of(int m) {
    const int n = __popc(m);
    return (n == 0 || n == 4) ? 0 : (n == 2 ? 2 : 1);
}

__device__ __forceinline__ float pick(const Cube &q, int c) {
    float v = q.f[0];
#pragma unroll
    for (int b = 1; b < 8; ++b) v = c == b ? q.f[b] : v;
    return v;
}

// The crossing of the edge between corners u and w, from the lower grid index
// (the lower corner code: indices grow with z, then y, then x) to the higher.
__device__ __forceinline__ void edge_point(const Cube &q, const Grid3 &g, int u, int w, float iso, float *out) {
    if (u > w) {
        const int t = u;
        u = w;
        w = t;
    }
    const float fu = pick(q, u), fw = pick(q, w);
    const float t = __fdiv_rn(__fsub_rn(iso, fu), __fsub_rn(fw, fu));
    const int at[3] = {q.i, q.j, q.k};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float pu = __fadd_rn(g.o[a], __fmul_rn(g.h, (float)(at[a] + ((u >> a) & 1))));
        const float pw = __fadd_rn(g.o[a], __fmul_rn(g.h, (float)(at[a] + ((w >> a) & 1))));
        out[a] = __fadd_rn(pu, __fmul_rn(t, __fsub_rn(pw, pu)));
    }
}

// Prefix sums without scratch beside the array: block b owns the kScanTile
// elements from b kScanTile on and writes the inclusive sums inside its tile,
// each one place up (a[i + 1] = sum of the tile's elements up to i; a[0] = 0).
// k_scan_tiles then makes the sums at the tiles' ends global, and a reader adds
// the tile's base to the places between them (tile_prefix).  One block scanning
// all elements took 3.6 ms for 2.1 M cubes.
constexpr int kScanThreads = 512;
constexpr int kScanPer = kScanTile / kScanThreads;

__device__ __forceinline__ int64_t tile_prefix(const int64_t *a, int64_t i) {
    const int64_t b = i & ~(int64_t)(kScanTile - 1);
    return i == b ? a[i] : a[b] + a[i];
}

__device__ __forceinline__ long long block_iscan_i64(long long v, long long *tmp, long long *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) tmp[warp] = v;
    __syncthreads();
    if (warp == 0) {
        long long w = lane < nw ? tmp[lane] : 0ll;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        tmp[lane] = w;
    }
    __syncthreads();
    *total = tmp[nw - 1];
    v += warp ? tmp[warp - 1] : 0ll;
    __syncthreads();
    return v;
}

// The tile sums of element values get(i), i < n, by one block per tile: a
// thread's values of all rounds first, their warp scans, then one scan of the
// rounds' and warps' totals (two barriers a tile).
template <typename F>
__device__ __forceinline__ void scan_tile(int64_t n, int64_t *a, F get) {
    constexpr int NW = kScanThreads / 32, N = NW * kScanPer;
    static_assert(N % 32 == 0, "whole warps of totals");
    __shared__ long long tot[N];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t base = blockIdx.x * (int64_t)kScanTile;
    if (blockIdx.x == 0 && threadIdx.x == 0) a[0] = 0;
    long long v[kScanPer];
#pragma unroll
    for (int r = 0; r < kScanPer; ++r) {
        const int64_t i = base + r * kScanThreads + threadIdx.x;
        v[r] = i < n ? get(i) : 0ll;
    }
#pragma unroll
    for (int r = 0; r < kScanPer; ++r) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long t = __shfl_up_sync(0xffffffffu, v[r], o);
            if (lane >= o) v[r] += t;
        }
        if (lane == 31) tot[r * NW + warp] = v[r];
    }
    __syncthreads();
    if (warp == 0) {
        long long carry = 0;
        for (int q = 0; q < N; q += 32) {
            const long long own = tot[q + lane];
            long long inc = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            tot[q + lane] = carry + inc - own;
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kScanPer; ++r) {
        const int64_t i = base + r * kScanThreads + threadIdx.x;
        if (i < n) a[i + 1] = tot[r * NW + warp] + v[r];
    }
}

// One block: the sums at the tiles' ends (and at n) become global ones.
__global__ void __launch_bounds__(1024) k_scan_tiles(int64_t *a, int64_t n) {
    pdl_wait();
    pdl_trigger();
    __shared__ long long tmp[32];
    const int64_t tiles = (n + kScanTile - 1) / kScanTile;
    long long carry = 0;
    for (int64_t t0 = 0; t0 < tiles; t0 += blockDim.x) {
        const int64_t t = t0 + threadIdx.x, at = min((t + 1) * (int64_t)kScanTile, n);
        long long total;
        const long long v = block_iscan_i64(t < tiles ? a[at] : 0ll, tmp, &total);
        if (t < tiles) a[at] = carry + v;
        carry += total;
    }
}

__global__ void __launch_bounds__(kScanThreads) k_mt_count(const float *f, Grid3 g, float iso, int64_t ncubes,
                                                           int64_t *off) {
    pdl_wait();
    pdl_trigger();
    scan_tile(ncubes, off, [&](int64_t c) {
        const int in = inside(cube_at(f, g, c), iso);
        int n = 0;
        if (in != 0 && in != 255) {
#pragma unroll
            for (int t = 0; t < 6; ++t) n += tris_of(tet_mask(in, t));
        }
        return (long long)n;
    });
}

// A block first lists its crossed cubes (about one in thirty of a surface's
// grid), then a thread takes one tetrahedron of one listed cube, so that warps
// are full of them; cubes taken where they lie left a few lanes of each warp
// working (61 us for 2.1 M cubes, now 31).
constexpr int kMtThreads = 256;
__global__ void __launch_bounds__(kMtThreads) k_mt_write(const float *f, Grid3 g, float iso, int64_t ncubes,
                                                         const int64_t *off, float *tri) {
    __shared__ uint16_t s_cube[kMtThreads];
    __shared__ uint8_t s_in[kMtThreads];
    __shared__ uint32_t tmp[33];
    const int64_t base = blockIdx.x * (int64_t)kMtThreads, mine = base + threadIdx.x;
    int in = 0;
    if (mine < ncubes) in = inside(cube_at(f, g, mine), iso);
    const bool crossed = in != 0 && in != 255;
    uint32_t n;
    const uint32_t at = block_exscan(crossed, tmp, &n);
    if (crossed) {
        s_cube[at] = (uint16_t)threadIdx.x;
        s_in[at] = (uint8_t)in;
    }
    __syncthreads();
    for (uint32_t w = threadIdx.x; w < 6 * n; w += kMtThreads) {
        const uint32_t a = w / 6, k = w - 6 * a;
        const int all = s_in[a], m = tet_mask(all, k), nin = __popc(m);
        if (nin == 0 || nin == 4) continue;
        const int64_t c = base + s_cube[a];
        int64_t o = tile_prefix(off, c);
        for (uint32_t b = 0; b < k; ++b) o += tris_of(tet_mask(all, b));
        float *t = tri + 9 * o;
        const Cube q = cube_at(f, g, c);
        const int *v = c_tets[k];
        if (nin != 2) {
            const int l = __ffs(nin == 1 ? m : ~m & 15) - 1;  // the lone vertex
#pragma unroll
            for (int e = 0; e < 3; ++e) edge_point(q, g, v[l], v[e + (e >= l)], iso, t + 3 * e);
        } else {
            const int A = __ffs(m) - 1, B = 31 - __clz(m), C = __ffs(~m & 15) - 1, D = 31 - __clz(~m & 15);
            float ac[3], ad[3], bd[3], bc[3];
            edge_point(q, g, v[A], v[C], iso, ac);
            edge_point(q, g, v[A], v[D], iso, ad);
            edge_point(q, g, v[B], v[D], iso, bd);
            edge_point(q, g, v[B], v[C], iso, bc);
#pragma unroll
            for (int a3 = 0; a3 < 3; ++a3) {
                t[a3] = ac[a3];
                t[3 + a3] = ad[a3];
                t[6 + a3] = bd[a3];
                t[9 + a3] = ac[a3];
                t[12 + a3] = bd[a3];
                t[15 + a3] = bc[a3];
            }
        }
    }
}

// Cross product of the triangle's edges, float, fixed operation order.
__device__ __forceinline__ void tri_cross(const float *t, float &cx, float &cy, float &cz) {
    const float ux = __fsub_rn(t[3], t[0]), uy = __fsub_rn(t[4], t[1]), uz = __fsub_rn(t[5], t[2]);
    const float vx = __fsub_rn(t[6], t[0]), vy = __fsub_rn(t[7], t[1]), vz = __fsub_rn(t[8], t[2]);
    cx = __fsub_rn(__fmul_rn(uy, vz), __fmul_rn(uz, vy));
    cy = __fsub_rn(__fmul_rn(uz, vx), __fmul_rn(ux, vz));
    cz = __fsub_rn(__fmul_rn(ux, vy), __fmul_rn(uy, vx));
}

__device__ __forceinline__ float norm3(float cx, float cy, float cz) {
    return __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(cx, cx), __fmul_rn(cy, cy)), __fmul_rn(cz, cz)));
}

// Triangle areas quantised to 64-bit integers (unit 2^-40): exact prefix sums,
// in scan_tile's form.
__global__ void __launch_bounds__(kScanThreads) k_area_q(const float *tri, int64_t ntri, int64_t *cum) {
    pdl_wait();
    pdl_trigger();
    scan_tile(ntri, cum, [&](int64_t k) {
        float cx, cy, cz;
        tri_cross(tri + 9 * k, cx, cy, cz);
        const float a = __fmul_rn(0.5f, norm3(cx, cy, cz));
        return (long long)__double2ll_rn(__dmul_rn((double)a, 1099511627776.0));
    });
}

__global__ void k_sample(const float *tri, int64_t ntri, const int64_t *cum, const double *u, int64_t ns, float *pts,
                         float *nrm) {
    const uint64_t total = (uint64_t)cum[ntri];
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns; s += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t target = (uint64_t)__dmul_rn(u[3 * s], (double)total);
        int64_t lo = 0, hi = ntri;  // the k with cum[k] <= target < cum[k + 1]
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) / 2;
            if ((uint64_t)tile_prefix(cum, mid) <= target) lo = mid; else hi = mid;
        }
        const float *t = tri + 9 * lo;
        const float r = __fsqrt_rn(__double2float_rn(u[3 * s + 1])), w = __double2float_rn(u[3 * s + 2]);
        const float ca = __fsub_rn(1.0f, r), cb = __fmul_rn(r, __fsub_rn(1.0f, w)), cc = __fmul_rn(r, w);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            pts[3 * s + a] = __fadd_rn(__fadd_rn(__fmul_rn(ca, t[a]), __fmul_rn(cb, t[3 + a])), __fmul_rn(cc, t[6 + a]));
        float cx, cy, cz;
        tri_cross(t, cx, cy, cz);
        const float len = norm3(cx, cy, cz);
        nrm[3 * s] = __fdiv_rn(cx, len);
        nrm[3 * s + 1] = __fdiv_rn(cy, len);
        nrm[3 * s + 2] = __fdiv_rn(cz, len);
    }
}

// ---------------------------------------------------------------- nearest points
// The nearest point of Q for every point of P, its float squared distance in a
// fixed operation order, ties to the lowest index: the value does not depend on
// how Q is searched.  Sets of kNnMin points and more are searched through a
// grid of 8^levels cells over their box, cells in Morton order, so that every
// node of the implied octree is a contiguous range of cells and of points; a
// query descends nearest child first and leaves out nodes whose (rounded down)
// distance is above the best.  All pairs took 10.5 ms for two sets of 10^5
// points, this 0.25 ms with the grids' making.  Smaller sets are streamed through shared memory.
constexpr int kNnThreads = 256;
// From so many points on a set gets a grid: the metrics of two sets of 1000 take
// 66 us streamed and 94 by grids, of 2000 77 and 80, of 5000 131 and 92 (the five
// launches that make a grid cost about 15).
constexpr int64_t kNnMin = 1024;
constexpr int kNnMaxLevels = 8;
constexpr int kNnLeaf = 16;  // nodes of so few points are not split further (8, 16, 32: 253, 270, 263 us for 10^5)
// A set with more than 1 / kNnDense of its points in one cell is streamed as
// well: a far point stretches the box until a cluster lies in a few cells, and
// its queries would walk them point by point through the index.  Two sets of
// 10^5 points, each with one point at a hundred times the others' extent: 18.0 ms
// by cells, 8.8 streamed (all pairs at any time: 10.8 before the grid).  At ten
// times the extent (densest cell below 1 / 8) cells take 1.5 ms.
constexpr int64_t kNnDense = 8;

__device__ __forceinline__ float nn_d2(float px, float py, float pz, const float *q) {
    const float dx = __fsub_rn(px, q[0]), dy = __fsub_rn(py, q[1]), dz = __fsub_rn(pz, q[2]);
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// One set and its grid.  box: ordered keys of the least and the largest finite
// coordinate per axis, then the most points in one cell.
struct NnSet {
    const float *p;
    int64_t n;
    int levels;     // < 0: no grid
    uint32_t *end;  // per cell, after k_nn_fill: one past its last point
    uint32_t *idx;  // point indices by cell
    int *box;       // 7
};

struct NnFrame {
    float lo[3], size[3], inv[3], pad[3];
};

__device__ __forceinline__ int nn_key(float f) {
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}

// Cell edges, and a pad that covers the rounding of a point's cell and of a
// cell's faces.  A set without finite points has some frame; it does not matter.
__device__ __forceinline__ NnFrame nn_frame(const NnSet &s) {
    NnFrame f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int kl = s.box[a], kh = s.box[3 + a];
        const float lo = __int_as_float(kl >= 0 ? kl : kl ^ 0x7fffffff), hi = __int_as_float(kh >= 0 ? kh : kh ^ 0x7fffffff);
        f.lo[a] = lo;
        f.size[a] = (hi - lo) * exp2f((float)-s.levels);
        f.inv[a] = f.size[a] > 0.f ? 1.f / f.size[a] : 0.f;
        f.pad[a] = 1e-4f * f.size[a] + 4e-7f * (fabsf(lo) + fabsf(hi));
    }
    return f;
}

__device__ __forceinline__ uint32_t spread3(uint32_t v) {  // bits 0..9 to every third bit
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    return (v | (v << 2)) & 0x09249249u;
}

__device__ __forceinline__ uint32_t nn_cell(const NnFrame &f, int levels, const float *q) {
    uint32_t m = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float c = fminf(fmaxf((q[a] - f.lo[a]) * f.inv[a], 0.f), (float)((1 << levels) - 1));
        m |= spread3((uint32_t)c) << a;
    }
    return m;
}

struct NnSets {
    NnSet s[2];
};

// Cell counts to zero, boxes to empty.
__global__ void k_nn_clear(NnSets a) {
    pdl_wait();
    pdl_trigger();
    const NnSet &s = a.s[blockIdx.y];
    if (s.levels < 0) return;
    const int64_t cells = (int64_t)1 << (3 * s.levels);
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < cells; c += (int64_t)gridDim.x * blockDim.x)
        s.end[c] = 0u;
    if (blockIdx.x == 0 && threadIdx.x < 7)
        s.box[threadIdx.x] = threadIdx.x < 3 ? 0x7fffffff : (threadIdx.x < 6 ? (int)0x80000000 : 0);
}

__global__ void __launch_bounds__(256) k_nn_box(NnSets a) {
    pdl_wait();
    pdl_trigger();
    const NnSet &s = a.s[blockIdx.y];
    if (s.levels < 0) return;
    int lo[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, hi[3] = {(int)0x80000000, (int)0x80000000, (int)0x80000000};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < s.n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float v = s.p[3 * i + q];
            if (fabsf(v) < INFINITY) {
                lo[q] = min(lo[q], nn_key(v));
                hi[q] = max(hi[q], nn_key(v));
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        lo[q] = __reduce_min_sync(0xffffffffu, lo[q]);
        hi[q] = __reduce_max_sync(0xffffffffu, hi[q]);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&s.box[q], lo[q]);
            atomicMax(&s.box[3 + q], hi[q]);
        }
    }
}

// FILL = false: points per cell; true: their indices by cell (in any order
// within a cell), after which end[c] is one past the cell's last.
template <bool FILL>
__global__ void __launch_bounds__(256) k_nn_cells(NnSets a) {
    pdl_wait();
    pdl_trigger();
    const NnSet &s = a.s[blockIdx.y];
    if (s.levels < 0) return;
    const NnFrame f = nn_frame(s);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < s.n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t o = atomicAdd(&s.end[nn_cell(f, s.levels, s.p + 3 * i)], 1u);
        if (FILL) s.idx[o] = (uint32_t)i;
    }
}

// One block per set: counts become first positions.
__global__ void __launch_bounds__(1024) k_nn_scan(NnSets a) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t tmp[33];
    const NnSet &s = a.s[blockIdx.x];
    if (s.levels < 0) return;
    const int64_t cells = (int64_t)1 << (3 * s.levels);
    uint32_t carry = 0, most = 0;
    for (int64_t c0 = 0; c0 < cells; c0 += 4096) {
        const int64_t c = c0 + 4 * threadIdx.x;
        uint32_t v[4], sum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = c + k < cells ? s.end[c + k] : 0u;
            sum += v[k];
            most = max(most, v[k]);
        }
        uint32_t total, o = block_exscan(sum, tmp, &total) + carry;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (c + k < cells) s.end[c + k] = o;
            o += v[k];
        }
        carry += total;
    }
    most = __reduce_max_sync(0xffffffffu, most);
    if ((threadIdx.x & 31) == 0) atomicMax(&s.box[6], (int)most);
}

// Best point of the grid of Q for p, from (best, bi).
__device__ __forceinline__ void nn_search(const NnSet &s, const NnFrame &f, float px, float py, float pz, float &best,
                                          int64_t &bi) {
    uint32_t node[7 * kNnMaxLevels + 2];  // level << 27 | z << 18 | y << 9 | x
    float low[7 * kNnMaxLevels + 2];
    const float p[3] = {px, py, pz};
    int top = 0;
    node[0] = 0u;
    low[0] = 0.f;
    top = 1;
    while (top > 0) {
        --top;
        if (low[top] > best) continue;
        const uint32_t e = node[top];
        const int l = (int)(e >> 27), sh = 3 * (s.levels - l);
        const uint32_t x = e & 511u, y = (e >> 9) & 511u, z = (e >> 18) & 511u;
        const uint32_t m = spread3(x) | spread3(y) << 1 | spread3(z) << 2;
        const uint32_t c0 = m << sh, c1 = (m + 1u) << sh;
        const uint32_t b = c0 ? s.end[c0 - 1] : 0u, en = s.end[c1 - 1];
        if (b == en) continue;
        if (l == s.levels || en - b <= (uint32_t)kNnLeaf) {
            for (uint32_t k = b; k < en; ++k) {
                const uint32_t j = s.idx[k];
                const float d2 = nn_d2(px, py, pz, s.p + 3 * (int64_t)j);
                if (d2 < best || (d2 == best && (int64_t)j < bi)) {
                    best = d2;
                    bi = j;
                }
            }
            continue;
        }
        // children: distance per axis to the lower and the upper half
        const uint32_t at[3] = {x, y, z};
        float d[3][2];
        uint32_t nearc = 0;
        const float w = (float)(1 << (s.levels - l - 1));
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float half = w * f.size[a];
            const float e0 = f.lo[a] + (float)(2 * at[a]) * half, e1 = e0 + half, e2 = e1 + half;
            d[a][0] = fmaxf(fmaxf(e0 - f.pad[a] - p[a], p[a] - e1 - f.pad[a]), 0.f);
            d[a][1] = fmaxf(fmaxf(e1 - f.pad[a] - p[a], p[a] - e2 - f.pad[a]), 0.f);
            nearc |= (p[a] >= e1 ? 1u : 0u) << a;
        }
#pragma unroll
        for (int k = 7; k >= 0; --k) {  // the nearest child is taken next
            const uint32_t c = nearc ^ (uint32_t)k;
            const float dx = d[0][c & 1u], dy = d[1][(c >> 1) & 1u], dz = d[2][c >> 2];
            const float lb = (dx * dx + dy * dy + dz * dz) * 0.999999f;
            if (!(lb > best)) {
                node[top] = (uint32_t)(l + 1) << 27 | (2 * z + (c >> 2)) << 18 | (2 * y + ((c >> 1) & 1u)) << 9 |
                            (2 * x + (c & 1u));
                low[top++] = lb;
            }
        }
    }
}

// What a direction (points of P to set Q) needs: P's own grid, when it has
// one, gives the order in which its points are taken.
struct NnDir {
    NnSet P, Q;
    const float *nP, *nQ;
    float *best;     // per point of P: squared distance to the nearest of Q
    uint32_t *bi;    // and its index
    double *part;    // three doubles per block of k_nn_sums
};
struct NnDirs {
    NnDir d[2];
};

// Nearest points of both directions (blockIdx.y).  Points are taken in the
// order of their own grid, so the lanes of a warp walk about the same nodes (in
// the sampling order, 200 us a direction for 10^5 points each; now 155 for both).
__global__ void __launch_bounds__(kNnThreads) k_nearest(NnDirs a) {
    pdl_wait();
    pdl_trigger();
    __shared__ float sq[kNnThreads * 3];
    const NnDir &d = a.d[blockIdx.y];
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q - threadIdx.x >= d.P.n) return;
    const bool live = q < d.P.n;
    const int64_t i = live ? (d.P.levels >= 0 ? (int64_t)d.P.idx[q] : q) : 0;
    const float px = d.P.p[3 * i], py = d.P.p[3 * i + 1], pz = d.P.p[3 * i + 2];
    float best = INFINITY;
    int64_t bi = 0;
    if (d.Q.levels >= 0 && kNnDense * d.Q.box[6] <= d.Q.n) {
        if (live) nn_search(d.Q, nn_frame(d.Q), px, py, pz, best, bi);
    } else {
        for (int64_t j0 = 0; j0 < d.Q.n; j0 += kNnThreads) {
            __syncthreads();
            const int cnt = (int)min((int64_t)kNnThreads, d.Q.n - j0);
            for (int k = threadIdx.x; k < 3 * cnt; k += kNnThreads) sq[k] = d.Q.p[3 * j0 + k];
            __syncthreads();
            for (int k = 0; k < cnt; ++k) {
                const float d2 = nn_d2(px, py, pz, sq + 3 * k);
                if (d2 < best) {
                    best = d2;
                    bi = j0 + k;
                }
            }
        }
    }
    if (live) {
        d.best[i] = best;
        d.bi[i] = (uint32_t)bi;
    }
}

// Largest distance, sum of distances and sum of |n_P . n_Q| of a block's
// points, in a fixed order.
__global__ void __launch_bounds__(kNnThreads) k_nn_sums(NnDirs a) {
    pdl_wait();
    pdl_trigger();
    __shared__ double sm[3][32];
    const NnDir &D = a.d[blockIdx.y];
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i - threadIdx.x >= D.P.n) return;
    double d = 0.0, c = 0.0;
    if (i < D.P.n) {
        const float *p = D.nP + 3 * i, *q = D.nQ + 3 * (int64_t)D.bi[i];
        d = __dsqrt_rn((double)D.best[i]);
        c = fabs(__dadd_rn(__dadd_rn(__dmul_rn((double)p[0], (double)q[0]), __dmul_rn((double)p[1], (double)q[1])),
                           __dmul_rn((double)p[2], (double)q[2])));
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double m = d;
    for (int o = 16; o > 0; o >>= 1) {
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        d += __shfl_xor_sync(0xffffffffu, d, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (lane == 0) {
        sm[0][warp] = m;
        sm[1][warp] = d;
        sm[2][warp] = c;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
        m = fmax(m, sm[0][w]);
        d += sm[1][w];
        c += sm[2][w];
    }
    double *out = D.part + 3 * (int64_t)blockIdx.x;
    out[0] = m;
    out[1] = d;
    out[2] = c;
}

// One block per direction: the blocks' partials into red[3 x direction ..].
struct NnParts {
    const double *part[2];
    int64_t n[2];
    double *red;
};
__global__ void __launch_bounds__(1024) k_metric_sums(NnParts a) {
    pdl_wait();
    pdl_trigger();
    __shared__ double sm[3][32];
    const double *p = a.part[blockIdx.x];
    double m = 0.0, d = 0.0, c = 0.0;
    for (int64_t b = threadIdx.x; b < a.n[blockIdx.x]; b += blockDim.x) {
        m = fmax(m, p[3 * b]);
        d += p[3 * b + 1];
        c += p[3 * b + 2];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        d += __shfl_xor_sync(0xffffffffu, d, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (lane == 0) {
        sm[0][warp] = m;
        sm[1][warp] = d;
        sm[2][warp] = c;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
        m = fmax(m, sm[0][w]);
        d += sm[1][w];
        c += sm[2][w];
    }
    double *out = a.red + 3 * blockIdx.x;
    out[0] = m;
    out[1] = d;
    out[2] = c;
}

// Inverse of Eq. 3-10 on the branch S >= m: S = m + sqrt(-ln(t / 2) / h)
// (t >= 2 maps to m, t <= 0 to +inf).
__global__ void k_denormalize(const float *t, float *S, int64_t n, const double *mh) {
    const double m = mh[0], h = mh[1];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = (double)t[i];
        double s;
        if (v >= 2.0) s = m;
        else if (v <= 0.0) s = INFINITY;
        else s = m + sqrt(-log(v * 0.5) / h);
        S[i] = (float)s;
    }
}

__global__ void k_scatter(const float *src, const uint32_t *idx, float *dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[idx[i]] = src[i];
}

int blocks_for(int64_t n) {
    int64_t b = (n + 255) / 256;
    return (int)(b < 1 ? 1 : (b > 152 * 32 ? 152 * 32 : b));
}

}  // namespace

extern "C" int serbf_marching_tets(const float *f, const int32_t dims[3], const float origin[3], float h, float iso,
                                   float *tri, int64_t cap, int64_t *ntri, int64_t *scratch, void *stream) {
    SERBF_TRACE();
    if (!f || !dims || !origin || !ntri || !scratch || !(h > 0.f)) return SERBF_EINVAL;
    if (dims[0] < 2 || dims[1] < 2 || dims[2] < 2 || (cap > 0 && !tri)) return SERBF_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    Grid3 g{dims[0], dims[1], dims[2], {origin[0], origin[1], origin[2]}, h};
    const int64_t ncubes = (int64_t)(dims[0] - 1) * (dims[1] - 1) * (dims[2] - 1);
    launch_pdl(k_mt_count, dim3((unsigned)((ncubes + kScanTile - 1) / kScanTile)), dim3(kScanThreads), 0, s, f, g, iso,
               ncubes, scratch);
    launch_pdl(k_scan_tiles, dim3(1), dim3(1024), 0, s, scratch, ncubes);
    SERBF_CHECK_LAUNCH();
    int64_t n = 0;
    if (cudaMemcpyAsync(&n, scratch + ncubes, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return SERBF_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
    *ntri = n;
    if (n > cap) return SERBF_ECAPACITY;
    k_mt_write<<<(unsigned)((ncubes + kMtThreads - 1) / kMtThreads), kMtThreads, 0, s>>>(f, g, iso, ncubes, scratch, tri);
    SERBF_CHECK_LAUNCH();
    return cudaStreamSynchronize(s) == cudaSuccess ? SERBF_OK : SERBF_ECUDA;
}

extern "C" int serbf_sample_surface(const float *tri, int64_t ntri, const double *u, int64_t ns, float *pts, float *nrm,
                                    int64_t *scratch, void *stream) {
    SERBF_TRACE();
    if (!tri || ntri < 1 || !u || ns < 0 || (ns > 0 && (!pts || !nrm)) || !scratch) return SERBF_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    launch_pdl(k_area_q, dim3((unsigned)((ntri + kScanTile - 1) / kScanTile)), dim3(kScanThreads), 0, s, tri, ntri, scratch);
    launch_pdl(k_scan_tiles, dim3(1), dim3(1024), 0, s, scratch, ntri);
    SERBF_CHECK_LAUNCH();
    int64_t total = 0;
    if (cudaMemcpyAsync(&total, scratch + ntri, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return SERBF_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
    if (total <= 0) return SERBF_EINVAL;
    if (ns > 0) k_sample<<<blocks_for(ns), 256, 0, s>>>(tri, ntri, scratch, u, ns, pts, nrm);
    SERBF_CHECK_LAUNCH();
    return cudaStreamSynchronize(s) == cudaSuccess ? SERBF_OK : SERBF_ECUDA;
}

extern "C" int serbf_surface_metrics(const float *A, const float *nA, int64_t na, const float *B, const float *nB,
                                     int64_t nb, double out[3], double *scratch, void *stream) {
    SERBF_TRACE();
    if (!A || !nA || !B || !nB || na < 1 || nb < 1 || !out || !scratch) return SERBF_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    // scratch (16 bytes per point and 48): the six results last; from the start
    // 8 bytes per point for the nearest points, the blocks' partials (a set of
    // one block writes its result in place), then per grid its box, cells and
    // indices -- at most 8 + 24 / 256 + 2 + 4 bytes per point and 32
    double *red = scratch + 2 * (na + nb), *next = scratch + na + nb;
    float *best = reinterpret_cast<float *>(scratch);
    NnDirs dirs{};
    NnParts parts{};
    parts.red = red;
    const float *pts[2] = {A, B}, *nrm[2] = {nA, nB};
    const int64_t n[2] = {na, nb};
    NnSets sets{};
    for (int d = 0; d < 2; ++d) {
        parts.n[d] = (n[d] + kNnThreads - 1) / kNnThreads;
        parts.part[d] = parts.n[d] > 1 ? next : red + 3 * d;
        if (parts.n[d] > 1) next += 3 * parts.n[d];
    }
    uint32_t *word = reinterpret_cast<uint32_t *>(next);
    bool grids = false;
    for (int d = 0; d < 2; ++d) {
        NnSet &q = sets.s[d];
        q.p = pts[d];
        q.n = n[d];
        q.levels = -1;
        if (n[d] < kNnMin || n[d] > 0x7fffffffll) continue;
        q.levels = 3;
        while (q.levels < kNnMaxLevels && ((int64_t)2 << (3 * q.levels + 3)) <= n[d]) ++q.levels;
        q.box = reinterpret_cast<int *>(word);
        q.end = word + 8;
        q.idx = q.end + ((int64_t)1 << (3 * q.levels));
        word = q.idx + n[d];
        grids = true;
    }
    for (int d = 0; d < 2; ++d) {
        dirs.d[d] = NnDir{sets.s[d], sets.s[1 - d], nrm[d], nrm[1 - d], best,
                          reinterpret_cast<uint32_t *>(best + n[d]), const_cast<double *>(parts.part[d])};
        best += 2 * n[d];
    }
    const int64_t most = na > nb ? na : nb;
    if (grids) {
        const dim3 grid((unsigned)blocks_for(most), 2);
        launch_pdl(k_nn_clear, grid, dim3(256), 0, s, sets);
        launch_pdl(k_nn_box, grid, dim3(256), 0, s, sets);
        launch_pdl(k_nn_cells<false>, grid, dim3(256), 0, s, sets);
        launch_pdl(k_nn_scan, dim3(2), dim3(1024), 0, s, sets);
        launch_pdl(k_nn_cells<true>, grid, dim3(256), 0, s, sets);
    }
    const dim3 each((unsigned)((most + kNnThreads - 1) / kNnThreads), 2);
    launch_pdl(k_nearest, each, dim3(kNnThreads), 0, s, dirs);
    launch_pdl(k_nn_sums, each, dim3(kNnThreads), 0, s, dirs);
    launch_pdl(k_metric_sums, dim3(2), dim3(1024), 0, s, parts);
    SERBF_CHECK_LAUNCH();
    double r[6];
    if (cudaMemcpyAsync(r, red, sizeof(r), cudaMemcpyDeviceToHost, s) != cudaSuccess) return SERBF_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
    out[0] = fmax(r[0], r[3]);
    out[1] = r[1] / (2.0 * (double)na) + r[4] / (2.0 * (double)nb);
    out[2] = r[2] / (2.0 * (double)na) + r[5] / (2.0 * (double)nb);
    return SERBF_OK;
}

extern "C" int serbf_denormalize_sdf(const float *t, float *S, int64_t n, const double *mh_dev, void *stream) {
    if (n < 0 || (n > 0 && (!t || !S || !mh_dev))) return SERBF_EINVAL;
    if (n > 0) k_denormalize<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(t, S, n, mh_dev);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

extern "C" int serbf_scatter(const float *src, const uint32_t *idx, float *dst, int64_t n, void *stream) {
    if (n < 0 || (n > 0 && (!src || !idx || !dst))) return SERBF_EINVAL;
    if (n > 0) k_scatter<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(src, idx, dst, n);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}
