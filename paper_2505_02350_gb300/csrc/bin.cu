// Point binning (the data structure behind the support test of Eq. 3-15).
//
// Cells of edge h are grouped into super cells of sf^3 cells.  Points are
// radix-sorted by (super cell, cell within the super cell, original index), so
// every super cell -- and every cell -- is a contiguous range of binned
// points.  Each super cell's range is cut into 32-point tiles (one warp each);
// tiles never straddle a super cell, so they are full except the last one of
// each super cell, and a tile's bounding box is tight.
//
// Short launches, each started early behind its predecessor: keys with the first
// digit's histogram, then per 8-bit digit of the cell key a scatter, from the
// second digit on a histogram, and above 32 sort blocks a scan of its rows, the
// last scatter moving the points; then cells, super cells and tiles.  With d
// digits that is 3 + 2 d launches, or 3 + 3 d above 32 blocks: seven for 10 000
// samples in up to 65536 cells, twelve for 9.4 M points.  What bounds it is memory for large sets
// and launches for small ones.  It replaced scans by a single block and a
// serial walk per super cell: 2.1 M points took 576 us of kernels, now about
// 130; 10 000 points 130 us, now about 45.  Also the Sec. 3.4.2
// refinement entry point, which re-bins the grown training set.
#include <math.h>

#include <utility>

#include "common.cuh"

using namespace serbf;

namespace {

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortRounds = kSortTile / kSortThreads;        // elements per thread
constexpr int kSmallRounds = kSmallSortTile / kSortThreads;  // ... of a small set

// Histogram of one 8-bit digit of a block's tile, stored digit-major.
__device__ __forceinline__ void store_hist(const uint32_t *h, uint32_t *hist, int64_t nblk) {
    if (threadIdx.x < 256) hist[(int64_t)threadIdx.x * nblk + blockIdx.x] = h[threadIdx.x];
}

// Cell keys of a tile of points and the histogram of their lowest digit (the
// first radix pass takes the point's index as its value).
template <int ROUNDS>
__global__ void __launch_bounds__(kSortThreads) k_keys(const float *x, const float *y, const float *z, int64_t n,
                                                       serbf_grid g, int sf, int nsx, int nsy, uint32_t *keys,
                                                       uint32_t *hist, int64_t nblk, uint32_t *cell_max) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t h[256];
    if (threadIdx.x < 256) h[threadIdx.x] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) cell_max[0] = 0u;
    __syncthreads();
    // three exact divisions and three integer ones per point were most of the
    // launch (20 us for 2.1 M points): a product decides all but the points
    // next to a cell face
    const float inv = __frcp_rn(g.h);
    const bool pow2 = (sf & (sf - 1)) == 0;
    const int lg = 31 - __clz(sf);
    const int64_t start = (int64_t)blockIdx.x * (ROUNDS * kSortThreads);
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int64_t i = start + r * kSortThreads + threadIdx.x;
        if (i < n) {
            const int kx = cell_axis_by(x[i], g.origin[0], g.h, inv, g.n[0]);
            const int ky = cell_axis_by(y[i], g.origin[1], g.h, inv, g.n[1]);
            const int kz = cell_axis_by(z[i], g.origin[2], g.h, inv, g.n[2]);
            const uint32_t key = pow2 ? cell_key_pow2(kx, ky, kz, lg, nsx, nsy) : cell_key(kx, ky, kz, sf, nsx, nsy);
            keys[i] = key;
            atomicAdd(&h[key & 255u], 1u);
        }
    }
    __syncthreads();
    store_hist(h, hist, nblk);
}

template <int ROUNDS>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t *keys, int64_t n, int shift, uint32_t *hist,
                                                             int64_t nblk) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t h[256];
    if (threadIdx.x < 256) h[threadIdx.x] = 0u;
    __syncthreads();
    const int64_t start = (int64_t)blockIdx.x * (ROUNDS * kSortThreads);
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int64_t e = start + r * kSortThreads + threadIdx.x;
        if (e < n) atomicAdd(&h[(keys[e] >> shift) & 255u], 1u);
    }
    __syncthreads();
    store_hist(h, hist, nblk);
}

// One block per digit: its counts become exclusive prefixes over the sort
// blocks, its total goes to tot[digit].
__global__ void __launch_bounds__(256) k_radix_rows(uint32_t *hist, int64_t nblk, uint32_t *tot) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t tmp[33];
    uint32_t *row = hist + (int64_t)blockIdx.x * nblk;
    uint32_t carry = 0;
    for (int64_t b0 = 0; b0 < nblk; b0 += 256) {
        const int64_t b = b0 + threadIdx.x;
        uint32_t sum;
        const uint32_t off = block_exscan(b < nblk ? row[b] : 0u, tmp, &sum);
        if (b < nblk) row[b] = carry + off;
        carry += sum;
    }
    if (threadIdx.x == 0) tot[blockIdx.x] = carry;
}

// Where the last radix pass puts the sorted points instead of the values.
struct PermOut {
    const float *x, *y, *z;
    uint32_t *perm;
    float *xb, *yb, *zb;
};

// Stable scatter of one tile by one digit.  A warp owns 256 consecutive
// elements, so ranks come from ballots and the warp's own running digit
// counts, without a block barrier per round; one scan over the warps then
// places them (a barrier for each of 16 rounds of 256 elements took 18 us for
// 10 000 points, this takes about 6).  vin == nullptr: the values are the
// indices.  tot == nullptr: few blocks, each sums the histograms itself.
template <bool LAST, int ROUNDS>
__global__ void __launch_bounds__(kSortThreads) k_radix_scatter(const uint32_t *kin, const uint32_t *vin, uint32_t *kout,
                                                                uint32_t *vout, int64_t n, int shift,
                                                                const uint32_t *hist, int64_t nblk, const uint32_t *tot,
                                                                PermOut o) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t wcnt[kSortWarps][256];
    __shared__ uint32_t tmp[33];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = tid; k < kSortWarps * 256; k += kSortThreads) (&wcnt[0][0])[k] = 0u;
    uint32_t total = 0, before = 0;
    if (tid < 256) {
        const uint32_t *row = hist + (int64_t)tid * nblk;
        if (tot) {
            total = tot[tid];
            before = row[blockIdx.x];
        } else {
            for (int b = 0; b < (int)nblk; ++b) {
                const uint32_t v = row[b];
                total += v;
                before += b < (int)blockIdx.x ? v : 0u;
            }
        }
    }
    const uint32_t base = block_exscan(total, tmp, nullptr) + before;  // barriers: wcnt is clear
    const int64_t e0 = (int64_t)blockIdx.x * (ROUNDS * kSortThreads) + warp * (ROUNDS * 32) + lane;
    uint32_t key[ROUNDS], rank[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) key[r] = e0 + 32 * r < n ? kin[e0 + 32 * r] : 0u;
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const uint32_t d = e0 + 32 * r < n ? (key[r] >> shift) & 255u : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t ahead = __popc(peers & ((1u << lane) - 1u));
        const uint32_t c = d < 256u ? wcnt[warp][d] : 0u;
        __syncwarp();
        if (ahead == 0 && d < 256u) wcnt[warp][d] = c + __popc(peers);
        __syncwarp();
        rank[r] = c + ahead;
    }
    __syncthreads();
    if (tid < 256) {
        uint32_t run = base;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) {
            const uint32_t c = wcnt[w][tid];
            wcnt[w][tid] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const int64_t e = e0 + 32 * r;
        if (e < n) {
            const uint32_t val = vin ? vin[e] : (uint32_t)e;
            const uint32_t pos = wcnt[warp][(key[r] >> shift) & 255u] + rank[r];
            kout[pos] = key[r];
            if (LAST) {
                o.perm[pos] = val;
                o.xb[pos] = o.x[val];
                o.yb[pos] = o.y[val];
                o.zb[pos] = o.z[val];
            } else {
                vout[pos] = val;
            }
        }
    }
}

// First binned point of every cell (a binary search of the sorted keys per
// cell: no counting atomics, no scan), and the most points in one cell (bounds
// the points in a ball).
__global__ void __launch_bounds__(256) k_cells(const uint32_t *keys, int64_t n, int64_t ncp, uint32_t *cell_start,
                                               uint32_t *cell_max) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t first[257];
    const int64_t c = blockIdx.x * (int64_t)256 + threadIdx.x;
    auto search = [&](int64_t k) {
        int64_t lo = 0, hi = n;  // first position with a key >= k
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if ((int64_t)keys[mid] < k) lo = mid + 1; else hi = mid;
        }
        return (uint32_t)lo;
    };
    if (c <= ncp) {
        const uint32_t f = search(c);
        first[threadIdx.x] = f;
        cell_start[c] = f;
        if (threadIdx.x == 255 && c < ncp) first[256] = search(c + 1);
    }
    __syncthreads();
    uint32_t cnt = c < ncp ? first[threadIdx.x + 1] - first[threadIdx.x] : 0u;
    cnt = __reduce_max_sync(0xffffffffu, cnt);
    if ((threadIdx.x & 31) == 0 && cnt) atomicMax(cell_max, cnt);
}

// One block: tiles and forward work items (both sets) of every super cell,
// numbered in super-cell order; out = {tiles, items of set 0, of set 1, most
// tiles in one super cell}.  Also clears the forward's scheduling state (no
// mean cost yet: the first forward files every item in the same class).  The
// block's passes over the super cells bound it, one barrier each and the next
// pass's loads ahead (three scans of three barriers each took 163 us for 97 336).
__global__ void __launch_bounds__(1024) k_supers(const uint32_t *cell_start, int nsuper, int cps, uint32_t *stile,
                                                 ItemSet two, ItemSet four, uint32_t *out, uint32_t *arrived) {
    pdl_wait();
    pdl_trigger();
    __shared__ uint32_t s_sum[2][3][32];  // per warp: tiles and items of either set
    __shared__ uint32_t s_max;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_max = 0u;
    if (threadIdx.x < 4) two.sched[threadIdx.x] = four.sched[threadIdx.x] = 0u;
    if (threadIdx.x < 2) two.total[threadIdx.x] = four.total[threadIdx.x] = 0ull;
    auto tiles_of = [&](int s) {
        if (s >= nsuper) return 0u;
        return (cell_start[(int64_t)(s + 1) * cps] - cell_start[(int64_t)s * cps] + kTile - 1) / kTile;
    };
    uint32_t base[3] = {0u, 0u, 0u}, mx = 0, next = tiles_of(threadIdx.x);
    int buf = 0;
    for (int s0 = 0; s0 < nsuper; s0 += blockDim.x, buf ^= 1) {
        const int s = s0 + threadIdx.x;
        const uint32_t nt = next, v[3] = {nt, (nt + 1) / 2, (nt + kMostTiles - 1) / kMostTiles};
        next = tiles_of(s + blockDim.x);
        mx = max(mx, nt);
        uint32_t inc[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            inc[k] = warp_iscan(v[k]);
            if (lane == 31) s_sum[buf][k][warp] = inc[k];
        }
        __syncthreads();  // the other buffer is written next: one barrier a pass
        uint32_t at[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t own = s_sum[buf][k][lane], to = warp_iscan(own);
            at[k] = base[k] + __shfl_sync(0xffffffffu, to - own, warp) + inc[k] - v[k];
            base[k] += __shfl_sync(0xffffffffu, to, 31);
        }
        if (s < nsuper) {
            stile[s] = at[0];
            two.super0[s] = at[1];
            four.super0[s] = at[2];
        }
    }
    __syncthreads();
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_max, mx);
    __syncthreads();
    if (threadIdx.x == 0) {
        stile[nsuper] = out[0] = base[0];
        two.super0[nsuper] = out[1] = base[1];
        four.super0[nsuper] = out[2] = base[2];
        out[3] = s_max;
        *arrived = 0u;
    }
}

__device__ __forceinline__ void warp_box(float x, float y, float z, bool v, float4 &lo, float4 &hi) {
    lo = make_float4(redux_min(v ? x : INFINITY), redux_min(v ? y : INFINITY), redux_min(v ? z : INFINITY), 0.f);
    hi = make_float4(redux_max(v ? x : -INFINITY), redux_max(v ? y : -INFINITY), redux_max(v ? z : -INFINITY), 0.f);
}

struct TilesArgs {
    const uint32_t *cell_start, *stile0;
    int nsuper, cps;
    uint32_t *tile_super, *tile_start;
    ItemSet two, four;
    const float *xb, *yb, *zb;
    float4 *tlo, *thi, *slo, *shi, *box;
    uint32_t *arrived;
};

__device__ __forceinline__ void grow(float4 &lo, float4 &hi, float4 a, float4 b) {
    lo = make_float4(fminf(lo.x, a.x), fminf(lo.y, a.y), fminf(lo.z, a.z), 0.f);
    hi = make_float4(fmaxf(hi.x, b.x), fmaxf(hi.y, b.y), fmaxf(hi.z, b.z), 0.f);
}

constexpr int kTilesThreads = 512;
constexpr int kTilesWarps = kTilesThreads / 32;
// Points per super cell up to which k_tiles takes many super cells a block: a
// block each costs a barrier, a fence and a counter, whatever it holds.  Whole
// binning, us, a block each / sixteen a block: 6000 points in 68 921 super cells
// 495 / 219, 300 000 in 97 336 965 / 344 (150 000 of them in one 908 / 463), 16,
// 32, 64 and 128 points in each of 27 000 386 / 209, 391 / 218, 460 / 293, 593 /
// 473, of 1000 105 / 97, 110 / 103, 129 / 118, 132 / 139.  While a block each fits
// the chip at once (512 super cells, those of a thin band: 93 / 101) it is taken.
constexpr int64_t kSparsePoints = 64;
constexpr int64_t kWaveBlocks = 2048 / kTilesThreads;  // blocks of k_tiles on an SM
constexpr uint32_t kAloneTiles = 4;  // a warp of the sparse form takes so many tiles by itself

__device__ __forceinline__ void put_item(const ItemSet &set, int s, uint32_t t, uint32_t k, uint32_t ps, uint32_t left,
                                         uint32_t tiles) {
    if (k % tiles) return;
    const uint32_t it = set.super0[s] + k / tiles;
    const uint4 r = make_uint4(t, (uint32_t)s, ps, (min(left, tiles * kTile) - 1u) | (it << 7));
    set.rec[it] = r;
    set.order[it] = r;
    set.cls[it] = 3;  // one class for all until a forward has measured them
}

// Tiles first, first + step, ... of super cell s, a warp at a time: their
// starts, boxes and work items; grows the box lo .. hi by theirs.
__device__ __forceinline__ void super_tiles(const TilesArgs &a, int s, uint32_t first, uint32_t step, int lane, float4 &lo,
                                            float4 &hi) {
    const uint32_t t0 = a.stile0[s], t1 = a.stile0[s + 1];
    const uint32_t p0 = a.cell_start[(int64_t)s * a.cps], pe = a.cell_start[(int64_t)(s + 1) * a.cps];
    for (uint32_t t = t0 + first; t < t1; t += step) {
        const uint32_t ps = p0 + (t - t0) * kTile, i = ps + lane;
        const bool v = i < pe;
        float4 tl, th;
        warp_box(v ? a.xb[i] : 0.f, v ? a.yb[i] : 0.f, v ? a.zb[i] : 0.f, v, tl, th);
        grow(lo, hi, tl, th);
        if (lane == 0) {
            a.tlo[t] = tl;
            a.thi[t] = th;
            a.tile_super[t] = (uint32_t)s;
            a.tile_start[t] = ps;
            put_item(a.two, s, t, t - t0, ps, pe - ps, 2u);
            put_item(a.four, s, t, t - t0, ps, pe - ps, (uint32_t)kMostTiles);
        }
    }
}

// One block per super cell, a warp per tile: the tile's start and bounding
// box, the work items (the first forward takes them in this order), the
// super cell's box (empty: +inf / -inf).  The last block unites the super
// cells' boxes (the box of every binned point).
// SPARSE: a block takes kTilesWarps super cells, a warp each, and all its warps
// together those of more than kAloneTiles tiles.
template <bool SPARSE>
__global__ void __launch_bounds__(kTilesThreads) k_tiles(TilesArgs a) {
    pdl_wait();
    pdl_trigger();
    constexpr int NW = kTilesWarps;
    __shared__ float4 wlo[NW], whi[NW];
    __shared__ bool s_many[NW];
    __shared__ bool s_last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // a block's super cells lie a grid apart, as dense ones lie side by side (a
    // thin band in 512 of them: 118 us with neighbours in a block, 108 so)
    const int s0 = blockIdx.x, ds = (int)gridDim.x, ns = SPARSE ? min(NW, (a.nsuper - s0 + ds - 1) / ds) : 1;
    const float4 none_lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    const float4 none_hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
    float4 lo = none_lo, hi = none_hi;
    if (SPARSE) {
        bool many = false;
        if (warp < ns) {
            const int s = s0 + warp * ds;
            many = a.stile0[s + 1] - a.stile0[s] > kAloneTiles;
            if (!many) {
                super_tiles(a, s, 0u, 1u, lane, lo, hi);
                if (lane == 0) {
                    a.slo[s] = lo;
                    a.shi[s] = hi;
                }
            }
        }
        if (lane == 0) s_many[warp] = many;
        __syncthreads();
    }
    for (int c = 0; c < ns; ++c) {
        if (SPARSE && !s_many[c]) continue;
        lo = none_lo;
        hi = none_hi;
        super_tiles(a, s0 + c * ds, (uint32_t)warp, (uint32_t)NW, lane, lo, hi);
        if (lane == 0) {
            wlo[warp] = lo;
            whi[warp] = hi;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < NW; ++w) grow(lo, hi, wlo[w], whi[w]);
            a.slo[s0 + c * ds] = lo;
            a.shi[s0 + c * ds] = hi;
        }
        if (SPARSE) __syncthreads();
    }
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(a.arrived, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    lo = none_lo;
    hi = none_hi;
    for (int q = threadIdx.x; q < a.nsuper; q += kTilesThreads) grow(lo, hi, __ldcg(a.slo + q), __ldcg(a.shi + q));
    float4 l, h;
    const float4 b = hi;
    warp_box(lo.x, lo.y, lo.z, true, l, h);
    lo = l;
    warp_box(b.x, b.y, b.z, true, l, h);
    if (lane == 0) {
        wlo[warp] = lo;
        whi[warp] = h;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        lo = none_lo;
        hi = none_hi;
        for (int w = 0; w < NW; ++w) grow(lo, hi, wlo[w], whi[w]);
        a.box[0] = lo;
        a.box[1] = hi;
    }
}

__global__ void k_concat(float *dst, const float *src, int64_t n) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        dst[k] = src[k];
}

int gsz(int64_t n, int t) {
    int64_t b = (n + t - 1) / t;
    if (b < 1) b = 1;
    if (b > 152 * 64) b = 152 * 64;
    return (int)b;
}

}  // namespace

namespace serbf {

// Small sets are cut into more, smaller sort tiles (10 000 points are three
// tiles of 4096: too few blocks to hide anything); up to kDirectBlocks of them
// every block sums the histograms itself instead of a launch for it.
struct SortPlan {
    int64_t nblk;
    bool small;
};
static SortPlan sort_plan(int64_t n) {
    const bool small = n <= (int64_t)kDirectBlocks * kSmallSortTile;
    const int64_t tile = small ? kSmallSortTile : kSortTile;
    return {(n + tile - 1) / tile, small};
}

template <int ROUNDS>
static void sort_pass(uint32_t *k, uint32_t *v, uint32_t *ko, uint32_t *vo, int64_t n, int shift, uint32_t *hist,
                      int64_t nblk, bool hist_done, const PermOut *out, cudaStream_t s) {
    const dim3 grid((unsigned)nblk), block(kSortThreads);
    if (!hist_done) launch_pdl(k_radix_hist<ROUNDS>, grid, block, 0, s, k, n, shift, hist, nblk);
    uint32_t *tot = nblk > kDirectBlocks ? hist + 256 * nblk : nullptr;
    if (tot) launch_pdl(k_radix_rows, dim3(256), dim3(256), 0, s, hist, nblk, tot);
    if (out)
        launch_pdl(k_radix_scatter<true, ROUNDS>, grid, block, 0, s, k, v, ko, vo, n, shift, hist, nblk, tot, *out);
    else
        launch_pdl(k_radix_scatter<false, ROUNDS>, grid, block, 0, s, k, v, ko, vo, n, shift, hist, nblk, tot, PermOut{});
}

// The passes of a sort.  keyed: the first digit's histogram is there already
// and the values are the indices.  With a PermOut the last pass writes it
// instead of the values.
static int sort_passes(uint32_t **k, uint32_t **v, uint32_t **ktmp, uint32_t **vtmp, int64_t n, int bits, uint32_t *hist,
                       bool keyed, const PermOut *out, cudaStream_t s) {
    const SortPlan p = sort_plan(n);
    for (int shift = 0; shift < bits; shift += 8) {
        const bool done = keyed && shift == 0;
        const PermOut *o = shift + 8 >= bits ? out : nullptr;
        (p.small ? sort_pass<kSmallRounds> : sort_pass<kSortRounds>)(*k, done ? nullptr : *v, *ktmp, *vtmp, n, shift, hist,
                                                                     p.nblk, done, o, s);
        std::swap(*k, *ktmp);
        std::swap(*v, *vtmp);
    }
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

int radix_sort_pairs(uint32_t **k, uint32_t **v, uint32_t **ktmp, uint32_t **vtmp, int64_t n, int bits,
                     uint32_t *hist, cudaStream_t s) {
    return sort_passes(k, v, ktmp, vtmp, n, bits, hist, false, nullptr, s);
}

}  // namespace serbf

extern "C" int serbf_bin_points(const float *x, const float *y, const float *z, int64_t n, const serbf_grid *grid,
                                uint32_t *perm, float *xb, float *yb, float *zb, serbf_workspace *ws,
                                void *stream) {
    SERBF_TRACE();
    if (!ws || ws->magic != kMagic || !grid || n < 0) return SERBF_EINVAL;
    if (n > 0 && (!x || !y || !z || !perm || !xb || !yb || !zb)) return SERBF_EINVAL;
    if (n > ws->sz.max_points) return SERBF_EINVAL;
    if (!(grid->h > 0.f) || grid->n[0] < 1 || grid->n[1] < 1 || grid->n[2] < 1) return SERBF_EINVAL;
    int64_t cells = (int64_t)grid->n[0] * grid->n[1] * grid->n[2];
    if (cells > ws->sz.max_cells) return SERBF_EINVAL;
    const int sf = ws->sz.super_factor, cps = sf * sf * sf;
    const int nsx = (grid->n[0] + sf - 1) / sf, nsy = (grid->n[1] + sf - 1) / sf, nsz = (grid->n[2] + sf - 1) / sf;
    const int64_t nsuper = (int64_t)nsx * nsy * nsz;
    if (nsuper > ws->max_supers) return SERBF_EINVAL;
    const int64_t ncp = nsuper * cps;  // cells including the padding of partial super cells
    cudaStream_t s = (cudaStream_t)stream;
    ws->grid = *grid;
    ws->sf = sf;
    ws->ns[0] = nsx;
    ws->ns[1] = nsy;
    ws->ns[2] = nsz;
    ws->nsuper = (int32_t)nsuper;
    ws->npoints = n;
    ws->binned = 0;

    uint32_t *kin = ws->keys0, *vin = ws->vals0, *kout = ws->keys1, *vout = ws->vals1;
    if (n > 0) {
        const SortPlan p = sort_plan(n);
        launch_pdl(p.small ? k_keys<kSmallRounds> : k_keys<kSortRounds>, dim3((unsigned)p.nblk), dim3(kSortThreads), 0, s, x,
                   y, z, n, *grid, sf, nsx, nsy, kin, ws->hist, p.nblk, ws->cell_max);
        int nbits = 1;
        while (nbits < 32 && (1ll << nbits) < ncp) ++nbits;
        const PermOut out{x, y, z, perm, xb, yb, zb};
        const int rc = sort_passes(&kin, &vin, &kout, &vout, n, nbits, ws->hist, true, &out, s);
        if (rc) return rc;
    } else if (cudaMemsetAsync(ws->cell_max, 0, sizeof(uint32_t), s) != cudaSuccess) {
        return SERBF_ECUDA;
    }
    launch_pdl(k_cells, dim3((unsigned)((ncp + 256) / 256)), dim3(256), 0, s, kin, n, ncp, ws->cell_start, ws->cell_max);
    uint32_t *out = ws->counters + 12;
    launch_pdl(k_supers, dim3(1), dim3(1024), 0, s, ws->cell_start, (int)nsuper, cps, ws->super_tile0, ws->items[0],
               ws->items[1], out, ws->counters);
    const bool sparse = n <= kSparsePoints * nsuper && nsuper > kWaveBlocks * (int64_t)ws->sm_count;
    launch_pdl(sparse ? k_tiles<true> : k_tiles<false>, dim3((unsigned)(sparse ? (nsuper + kTilesWarps - 1) / kTilesWarps : nsuper)),
               dim3(kTilesThreads), 0, s,
               TilesArgs{ws->cell_start, ws->super_tile0, (int)nsuper, cps, ws->tile_super, ws->tile_start, ws->items[0],
                         ws->items[1], xb, yb, zb, ws->tile_lo, ws->tile_hi, ws->sup_lo, ws->sup_hi, ws->field_box,
                         ws->counters});
    SERBF_CHECK_LAUNCH();
    uint32_t got[4];  // tiles, items of either set, most tiles in a super cell
    if (cudaMemcpyAsync(got, out, sizeof(got), cudaMemcpyDeviceToHost, s) != cudaSuccess) return SERBF_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
    if ((int64_t)got[0] > ws->max_tiles || got[1] >= (1u << 25)) return SERBF_ECAPACITY;  // item ids have 25 bits
    ws->ntiles = got[0];
    ws->items[0].n = got[1];
    ws->items[1].n = got[2];
    ws->max_chunks = (int32_t)((got[3] + kTile - 1) / kTile);
    ws->binned = 1;
    ws->unmeasured = 1;
    return SERBF_OK;
}

extern "C" int serbf_refine(float *x_all, float *y_all, float *z_all, float *t_all, float *s_all, int64_t n_old,
                            const float *x_new, const float *y_new, const float *z_new, const float *t_new,
                            const float *s_new, int64_t n_new, const serbf_grid *grid, uint32_t *perm, float *xb,
                            float *yb, float *zb, float *tb, float *sb, serbf_workspace *ws, void *stream) {
    SERBF_TRACE();
    if (!ws || ws->magic != kMagic || n_old < 0 || n_new < 0) return SERBF_EINVAL;
    if (!x_all || !y_all || !z_all || !t_all || !s_all || !tb || !sb) return SERBF_EINVAL;
    if (n_new > 0 && (!x_new || !y_new || !z_new || !t_new || !s_new)) return SERBF_EINVAL;
    int64_t n = n_old + n_new;
    if (n > ws->sz.max_points) return SERBF_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (n_new > 0) {
        k_concat<<<gsz(n_new, 256), 256, 0, s>>>(x_all + n_old, x_new, n_new);
        k_concat<<<gsz(n_new, 256), 256, 0, s>>>(y_all + n_old, y_new, n_new);
        k_concat<<<gsz(n_new, 256), 256, 0, s>>>(z_all + n_old, z_new, n_new);
        k_concat<<<gsz(n_new, 256), 256, 0, s>>>(t_all + n_old, t_new, n_new);
        k_concat<<<gsz(n_new, 256), 256, 0, s>>>(s_all + n_old, s_new, n_new);
        SERBF_CHECK_LAUNCH();
    }
    int rc = serbf_bin_points(x_all, y_all, z_all, n, grid, perm, xb, yb, zb, ws, stream);
    if (rc) return rc;
    rc = serbf_gather(t_all, perm, tb, n, stream);
    if (rc) return rc;
    return serbf_gather(s_all, perm, sb, n, stream);
}
