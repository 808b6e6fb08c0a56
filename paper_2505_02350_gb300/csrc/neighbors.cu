// Per-step rebuild of the kernel <-> point neighbour structure (Eq. 3-15,
// Eq. 3-15-1): per-kernel records and, per super cell, the list of kernels
// (ascending index) whose support may reach it.  The forward and the adjoint
// refine these lists against tight 32-point tile boxes and apply the exact
// support predicate per pair.  On request the explicit kernel-major and
// point-major CSR lists are produced from the same structure.
#include <math.h>
#include <string.h>

#include "common.cuh"
#include "order_rule.cuh"
#include "warps_rule.cuh"

using namespace serbf;

namespace {

// Per-kernel records.  kfwd: (c, r2), (Q11, Q22, Q33, a), (2Q12, 2Q13, 2Q23, l)
// with l the root of Q's largest eigenvalue and Q = log2(e) R^T D^2 R, so that exp(-||D R (v - c)||^2) = 2^(-dv^T Q dv);
// kbwd: (c, r2) and the rows of R with e_k = log2(e) d_k^2 in .w.
// R is the App. A matrix (entries r1..r9).
__device__ __forceinline__ void prep_kernels(const float *p, int cap, int m, float nle, float4 *kfwd, float4 *kbwd,
                                             int first, int stride) {
    for (int j = first; j < m; j += stride) {
        float cx = p[PCX * cap + j], cy = p[PCY * cap + j], cz = p[PCZ * cap + j];
        float d1 = p[PD1 * cap + j], d2 = p[PD2 * cap + j], d3 = p[PD3 * cap + j];
        float w = p[PW * cap + j];
        float sx, cxs, sy, cys, sz, czs;
        sincosf(p[PTX * cap + j], &sx, &cxs);
        sincosf(p[PTY * cap + j], &sy, &cys);
        sincosf(p[PTZ * cap + j], &sz, &czs);
        float R[9];
        R[0] = cxs * cys;
        R[1] = -czs * sx - sy * sz * cxs;
        R[2] = sx * sz - cxs * czs * sy;
        R[3] = cys * sx;
        R[4] = cxs * czs - sx * sy * sz;
        R[5] = -sz * cxs - czs * sx * sy;
        R[6] = sy;
        R[7] = cys * sz;
        R[8] = cys * czs;
        const float e[3] = {kLog2e * d1 * d1, kLog2e * d2 * d2, kLog2e * d3 * d3};
        float Q[3][3];
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b)
                Q[a][b] = fmaf(e[0] * R[a], R[b], fmaf(e[1] * R[3 + a], R[3 + b], e[2] * R[6 + a] * R[6 + b]));
        float r2 = support_r2(d1, d2, d3, nle);
        float aw = w * fabsf(w);
        kfwd[3 * j + 0] = make_float4(cx, cy, cz, r2);
        kfwd[3 * j + 1] = make_float4(Q[0][0], Q[1][1], Q[2][2], aw);
        kfwd[3 * j + 2] = make_float4(2.f * Q[0][1], 2.f * Q[0][2], 2.f * Q[1][2],
                                      sqrtf(fmaxf(e[0], fmaxf(e[1], e[2]))));
        kbwd[4 * j + 0] = make_float4(cx, cy, cz, r2);
        kbwd[4 * j + 1] = make_float4(R[0], R[1], R[2], e[0]);
        kbwd[4 * j + 2] = make_float4(R[3], R[4], R[5], e[1]);
        kbwd[4 * j + 3] = make_float4(R[6], R[7], R[8], e[2]);
    }
}

// One launch makes the order of so many items (the counters below hold 255 per
// thread of a block).
static_assert(kOrderDirectItems <= 128 * kOrderChunk, "items per thread of the one-launch order");

// The forward's heavy-first order for its next launch: a stable sort of the
// items by the cost class the last forward filed, descending, in one launch
// or two (order_direct) on the workspace's side stream (next to the neighbour
// rebuild).
// k_class_count: block b counts the classes of items [b kOrderChunk,
// (b + 1) kOrderChunk).  k_order_items: block b places the same items; a
// class starts after all heavier classes and after this class in earlier
// chunks, and the rank inside the chunk comes from ballots in item order.
__device__ __forceinline__ void class_count_body(const uint8_t *item_class, int64_t nitems, uint32_t *hist, int bx) {
    constexpr int NW = kOrderChunk / 32;
    __shared__ uint32_t s_wcnt[NW][kCostClasses];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)bx * kOrderChunk + threadIdx.x;
    const int cls = i < nitems ? (int)item_class[i] : -1;
#pragma unroll
    for (int c = 0; c < kCostClasses; ++c) {
        const unsigned bal = __ballot_sync(0xffffffffu, cls == c);
        if (lane == 0) s_wcnt[warp][c] = __popc(bal);
    }
    __syncthreads();
    if (threadIdx.x < kCostClasses) {
        uint32_t t = 0;
        for (int w = 0; w < NW; ++w) t += s_wcnt[w][threadIdx.x];
        hist[(size_t)bx * kCostClasses + threadIdx.x] = t;
    }
}

__global__ void __launch_bounds__(kOrderChunk) k_class_count(const uint8_t *item_class, int64_t nitems,
                                                             uint32_t *hist) {
    class_count_body(item_class, nitems, hist, blockIdx.x);
}

// hist == nullptr: the block counts the classes of all items itself.
__device__ __forceinline__ void order_items_body(const uint8_t *item_class, const uint32_t *hist,
                                                 const uint4 *item_rec, uint4 *order_rec, int64_t nitems, int bx) {
    constexpr int NW = kOrderChunk / 32;
    __shared__ uint32_t s_base[kCostClasses];      // first position of each class for this chunk
    __shared__ uint32_t s_tot[kCostClasses];
    __shared__ uint32_t s_wcnt[NW][kCostClasses];  // per warp: class counts, then offsets
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nchunks = (int)((nitems + kOrderChunk - 1) / kOrderChunk), b = bx;
    if (!hist) {
        if (threadIdx.x < kCostClasses) s_base[threadIdx.x] = s_tot[threadIdx.x] = 0u;
        __syncthreads();
        // four items at a time; eight 8-bit counters a thread (kOrderDirectItems
        // are 128 per thread)
        unsigned long long tot = 0ull, before = 0ull;
        for (int64_t i = 4 * (int64_t)threadIdx.x; i < nitems; i += 4 * kOrderChunk) {
            const uint32_t w = *reinterpret_cast<const uint32_t *>(item_class + i);
            unsigned long long c = 0ull;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (i + k < nitems) c += 1ull << (((w >> (8 * k)) & 7u) * 8);
            tot += c;
            if (i < (int64_t)b * kOrderChunk) before += c;
        }
#pragma unroll
        for (int c = 0; c < kCostClasses; ++c) {
            const uint32_t t = __reduce_add_sync(0xffffffffu, (uint32_t)(tot >> (8 * c)) & 255u);
            const uint32_t f = __reduce_add_sync(0xffffffffu, (uint32_t)(before >> (8 * c)) & 255u);
            if (lane == 0 && t) {
                atomicAdd(&s_tot[c], t);
                atomicAdd(&s_base[c], f);
            }
        }
    } else if (warp < kCostClasses) {
        // class totals and this class's count in earlier chunks: warp c handles class c
        uint32_t tot = 0, before = 0;
        for (int q = lane; q < nchunks; q += 32) {
            const uint32_t v = hist[(size_t)q * kCostClasses + warp];
            tot += v;
            before += q < b ? v : 0u;
        }
        tot = warp_sum(tot);
        before = warp_sum(before);
        if (lane == 0) {
            s_tot[warp] = tot;
            s_base[warp] = before;
        }
    }
    const int64_t i = (int64_t)b * kOrderChunk + threadIdx.x;
    const int cls = i < nitems ? (int)item_class[i] : -1;
    const uint4 r = i < nitems ? item_rec[i] : make_uint4(0u, 0u, 0u, 0u);
    uint32_t rank = 0;
#pragma unroll
    for (int c = 0; c < kCostClasses; ++c) {
        const unsigned bal = __ballot_sync(0xffffffffu, cls == c);
        if (cls == c) rank = __popc(bal & ((1u << lane) - 1u));
        if (lane == 0) s_wcnt[warp][c] = __popc(bal);
    }
    __syncthreads();
    if (threadIdx.x < kCostClasses) {
        const int c = threadIdx.x;
        uint32_t heavier = 0;  // classes are placed in descending order
        for (int q = c + 1; q < kCostClasses; ++q) heavier += s_tot[q];
        uint32_t run = heavier + s_base[c];
        for (int w = 0; w < NW; ++w) {
            const uint32_t v = s_wcnt[w][c];
            s_wcnt[w][c] = run;
            run += v;
        }
    }
    __syncthreads();
    if (cls >= 0) order_rec[s_wcnt[warp][cls] + rank] = r;
}

__global__ void __launch_bounds__(kOrderChunk) k_order_items(const uint8_t *item_class, const uint32_t *hist,
                                                             const uint4 *item_rec, uint4 *order_rec, int64_t nitems) {
    order_items_body(item_class, hist, item_rec, order_rec, nitems, blockIdx.x);
}

// Ascending list of the kernels that pass `hit`, by one block of
// kListThreads: a warp tests 128 consecutive candidates of each 1024 (four
// ballots), the warps' counts meet in shared memory (double-buffered: one
// barrier per 1024 candidates, where a block scan of every 256 took three: the
// first level of 9.4 M points and 16384 kernels 71 -> 62 us).
// Returns the count; entries beyond scap are not written.
constexpr int kListThreads = 256;
constexpr int kListWarps = kListThreads / 32;

template <typename F>
__device__ __forceinline__ uint32_t list_block(int m, uint32_t *out, int scap, F hit) {
    __shared__ uint32_t s_cnt[2][kListWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t count = 0;
    int buf = 0;
    for (int j0 = 0; j0 < m; j0 += 4 * kListThreads, buf ^= 1) {
        const int jw = j0 + 128 * warp + lane;
        unsigned bal[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) bal[r] = __ballot_sync(0xffffffffu, jw + 32 * r < m && hit(jw + 32 * r));
        if (lane == 0) s_cnt[buf][warp] = __popc(bal[0]) + __popc(bal[1]) + __popc(bal[2]) + __popc(bal[3]);
        __syncthreads();
        uint32_t at = count;
#pragma unroll
        for (int w = 0; w < kListWarps; ++w) {
            const uint32_t c = s_cnt[buf][w];
            at += w < warp ? c : 0u;
            count += c;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const uint32_t o = at + __popc(bal[r] & lt);
            if (((bal[r] >> lane) & 1u) && o < (uint32_t)scap) out[o] = (uint32_t)(jw + 32 * r);
            at += __popc(bal[r]);
        }
    }
    return count;
}

// Union of the boxes of the f x f x f super cells of block (cx, cy, cz).
__device__ __forceinline__ void block_box(const float4 *slo, const float4 *shi, int nsx, int nsy, int nsz, int cx, int cy,
                                          int cz, int f, float4 &lo, float4 &hi) {
    lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
    for (int dz = 0; dz < f; ++dz)
        for (int dy = 0; dy < f; ++dy)
            for (int dx = 0; dx < f; ++dx) {
                const int sx = f * cx + dx, sy = f * cy + dy, sz = f * cz + dz;
                if (sx >= nsx || sy >= nsy || sz >= nsz) continue;
                const int sc = (sz * nsy + sy) * nsx + sx;
                const float4 a = slo[sc], b = shi[sc];
                lo = make_float4(fminf(lo.x, a.x), fminf(lo.y, a.y), fminf(lo.z, a.z), 0.f);
                hi = make_float4(fmaxf(hi.x, b.x), fmaxf(hi.y, b.y), fmaxf(hi.z, b.z), 0.f);
            }
}

// The kernels of the parameter block whose support may reach a box (centre
// and r2 by the same float operations as the records).
__device__ __forceinline__ uint32_t list_params(const float *p, int cap, int m, float nle, float4 lo, float4 hi,
                                                uint32_t *out, int scap) {
    return list_block(m, out, scap, [&](int j) {
        const float r2 = support_r2(p[PD1 * cap + j], p[PD2 * cap + j], p[PD3 * cap + j], nle);
        return box_d2(p[PCX * cap + j], p[PCY * cap + j], p[PCZ * cap + j], lo, hi) < r2;
    });
}

// The same for a list that is filtered again with the records: the test is
// multiplied through by the least d^2 instead of dividing by it, with slack for
// the rounding of either side, so it keeps every kernel of list_params and
// perhaps one that just misses the box (that first level 62 -> 47 us).
__device__ __forceinline__ uint32_t list_params_about(const float *p, int cap, int m, float nle, float4 lo, float4 hi,
                                                      uint32_t *out, int scap) {
    const float lim = 1.00001f * nle;
    return list_block(m, out, scap, [&](int j) {
        const float d1 = p[PD1 * cap + j], d2 = p[PD2 * cap + j], d3 = p[PD3 * cap + j];
        float lam = d1 * d1;
        if (d2 * d2 < lam) lam = d2 * d2;
        if (d3 * d3 < lam) lam = d3 * d3;
        return box_d2(p[PCX * cap + j], p[PCY * cap + j], p[PCZ * cap + j], lo, hi) * lam < lim;
    });
}

// The per-step rebuild in one launch: blocks [0, nsuper) list, per super
// cell, every kernel whose support may reach its box; the remaining blocks
// write the per-kernel records.
__device__ __forceinline__ void rebuild_body(const float *p, int cap, const int32_t *m_dev, float nle, float4 *kfwd,
                                             float4 *kbwd, const float4 *slo, const float4 *shi, int nsuper,
                                             uint32_t *list, uint32_t *cnt, int scap, int32_t *status,
                                             long long *needed, int bx, int nbx) {
    const int m = *m_dev;
    const int s = bx;
    if (s >= nsuper) {
        prep_kernels(p, cap, m, nle, kfwd, kbwd, (s - nsuper) * blockDim.x + threadIdx.x,
                     (nbx - nsuper) * blockDim.x);
        return;
    }
    const float4 lo = slo[s], hi = shi[s];
    if (!(lo.x <= hi.x)) {
        if (threadIdx.x == 0) cnt[s] = 0;
        return;
    }
    const uint32_t count = list_params(p, cap, m, nle, lo, hi, list + (size_t)s * scap, scap);
    if (threadIdx.x == 0) {
        cnt[s] = count;
        if (count > (uint32_t)scap) {
            atomicOr(status, SERBF_FLAG_SUPER_LIST);
            atomicMax(needed + 0, (long long)count);
        }
    }
}

__global__ void __launch_bounds__(kListThreads) k_rebuild(const float *p, int cap, const int32_t *m_dev, float nle,
                                                          float4 *kfwd, float4 *kbwd, const float4 *slo, const float4 *shi,
                                                          int nsuper, uint32_t *list, uint32_t *cnt, int scap,
                                                          int32_t *status, long long *needed) {
    pdl_wait();
    pdl_trigger();
    rebuild_body(p, cap, m_dev, nle, kfwd, kbwd, slo, shi, nsuper, list, cnt, scap, status, needed, blockIdx.x,
                 gridDim.x);
}

// Rebuild in levels, for many super cells and kernels.  First launch: blocks
// [0, ncoarse) list, per block of f x f x f super cells (f = 2; 4 for the
// first of three levels), every kernel whose support may reach the union of
// their boxes (as k_rebuild does per super cell); the remaining blocks write
// the per-kernel records.
__device__ __forceinline__ void coarse_lists_body(const float *p, int cap, const int32_t *m_dev, float nle,
                                                  float4 *kfwd, float4 *kbwd, const float4 *slo, const float4 *shi,
                                                  int nsx, int nsy, int nsz, int ncoarse, uint32_t *list,
                                                  uint32_t *cnt, int scap, int bx, int nbx, int f) {
    __shared__ float4 s_lo, s_hi;
    const int m = *m_dev;
    const int c = bx;
    if (c >= ncoarse) {
        prep_kernels(p, cap, m, nle, kfwd, kbwd, (c - ncoarse) * blockDim.x + threadIdx.x,
                     (nbx - ncoarse) * blockDim.x);
        return;
    }
    if (threadIdx.x == 0) {
        const int ncx = (nsx + f - 1) / f, ncy = (nsy + f - 1) / f;
        block_box(slo, shi, nsx, nsy, nsz, c % ncx, (c / ncx) % ncy, c / (ncx * ncy), f, s_lo, s_hi);
    }
    __syncthreads();
    const float4 lo = s_lo, hi = s_hi;
    if (!(lo.x <= hi.x)) {
        if (threadIdx.x == 0) cnt[c] = 0;
        return;
    }
    const uint32_t count = list_params_about(p, cap, m, nle, lo, hi, list + (size_t)c * scap, scap);
    if (threadIdx.x == 0) cnt[c] = count;
}

__global__ void __launch_bounds__(kListThreads) k_coarse_lists(const float *p, int cap, const int32_t *m_dev, float nle,
                                                               float4 *kfwd, float4 *kbwd, const float4 *slo,
                                                               const float4 *shi, int nsx, int nsy, int nsz, int ncoarse,
                                                               uint32_t *list, uint32_t *cnt, int scap, int f) {
    pdl_wait();
    pdl_trigger();
    coarse_lists_body(p, cap, m_dev, nle, kfwd, kbwd, slo, shi, nsx, nsy, nsz, ncoarse, list, cnt, scap, blockIdx.x,
                      gridDim.x, f);
}

// Next levels: one block per parent (a block of super cells), one warp per
// child (2 x 2 x 2 of them).  The parent's candidates are fetched once for all
// eight children, 256 at a time, into shared memory; each warp keeps those
// that reach its child's box, tested with the records' centre and r2 (the
// values k_rebuild computes), 32 at a time and without a block scan.  A kernel
// that reaches a box reaches every box containing it, so the lists equal the
// one-level ones; a parent list that overflowed is not used (every kernel is
// tested).  With a block per child and a scan per 256 candidates the last two
// levels took 106 us of an epoch of 9.4 M points (32768 super cells), now 42.
// FINE: children are super cells, and their overflow is reported; otherwise
// they are blocks of 2 x 2 x 2 super cells.
struct ChildArgs {
    const int32_t *m_dev;
    const float4 *kfwd, *slo, *shi;
    int nsx, nsy, nsz;
    const uint32_t *plist, *pcnt;
    uint32_t *list, *cnt;
    int scap;
    int32_t *status;
    long long *needed;
};

template <bool FINE>
__device__ __forceinline__ void child_lists_body(const ChildArgs &a, int p) {
    __shared__ float4 s_k[kListThreads];
    __shared__ uint32_t s_j[kListThreads];
    static_assert(kListWarps == 8, "a warp per child");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    // grid of the children and of their parents
    const int nx = FINE ? a.nsx : (a.nsx + 1) >> 1, ny = FINE ? a.nsy : (a.nsy + 1) >> 1;
    const int nz = FINE ? a.nsz : (a.nsz + 1) >> 1;
    const int px = (nx + 1) >> 1, py = (ny + 1) >> 1;
    const int cx = 2 * (p % px) + (warp & 1), cy = 2 * ((p / px) % py) + ((warp >> 1) & 1), cz = 2 * (p / (px * py)) + (warp >> 2);
    const bool child = cx < nx && cy < ny && cz < nz;
    const int c = child ? (cz * ny + cy) * nx + cx : 0;
    float4 lo, hi;
    if (FINE) {
        lo = a.slo[c];
        hi = a.shi[c];
    } else {
        // a lane per super cell of the child
        const int sx = 2 * cx + (lane & 1), sy = 2 * cy + ((lane >> 1) & 1), sz = 2 * cz + ((lane >> 2) & 1);
        const bool in = child && sx < a.nsx && sy < a.nsy && sz < a.nsz;
        const int s = in ? (sz * a.nsy + sy) * a.nsx + sx : 0;
        lo = in ? a.slo[s] : make_float4(INFINITY, INFINITY, INFINITY, 0.f);
        hi = in ? a.shi[s] : make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            lo.x = fminf(lo.x, __shfl_xor_sync(0xffffffffu, lo.x, o));
            lo.y = fminf(lo.y, __shfl_xor_sync(0xffffffffu, lo.y, o));
            lo.z = fminf(lo.z, __shfl_xor_sync(0xffffffffu, lo.z, o));
            hi.x = fmaxf(hi.x, __shfl_xor_sync(0xffffffffu, hi.x, o));
            hi.y = fmaxf(hi.y, __shfl_xor_sync(0xffffffffu, hi.y, o));
            hi.z = fmaxf(hi.z, __shfl_xor_sync(0xffffffffu, hi.z, o));
        }
    }
    const bool any = child && lo.x <= hi.x;  // the child holds points
    const uint32_t pn = a.pcnt[p];
    const bool whole = pn > (uint32_t)a.scap;
    const int L = whole ? *a.m_dev : (int)pn;
    const uint32_t *src = a.plist + (size_t)p * a.scap;
    uint32_t *out = a.list + (size_t)c * a.scap;
    uint32_t count = 0;
    for (int q0 = 0; q0 < L; q0 += kListThreads) {
        __syncthreads();
        const int q = q0 + threadIdx.x;
        if (q < L) {
            const uint32_t j = whole ? (uint32_t)q : src[q];
            s_j[threadIdx.x] = j;
            s_k[threadIdx.x] = a.kfwd[3 * (size_t)j];
        }
        __syncthreads();
        if (!any) continue;
        const int n = min(kListThreads, L - q0);
        for (int b = 0; b < n; b += 32) {
            const float4 k = s_k[b + lane];
            const bool hit = b + lane < n && box_d2(k.x, k.y, k.z, lo, hi) < k.w;
            const unsigned bal = __ballot_sync(0xffffffffu, hit);
            const uint32_t o = count + __popc(bal & lt);
            if (hit && o < (uint32_t)a.scap) out[o] = s_j[b + lane];
            count += __popc(bal);
        }
    }
    if (child && lane == 0) {
        a.cnt[c] = count;
        if (FINE && count > (uint32_t)a.scap) {
            atomicOr(a.status, SERBF_FLAG_SUPER_LIST);
            atomicMax(a.needed + 0, (long long)count);
        }
    }
}

template <bool FINE>
__global__ void __launch_bounds__(kListThreads) k_child_lists(ChildArgs a) {
    pdl_wait();
    pdl_trigger();
    child_lists_body<FINE>(a, blockIdx.x);
}

// ---------------------------------------------------------------- batches of fields
// One field's neighbour rebuild for the batched epoch: the arguments of the
// single-field launches, and which form (one or two levels) it takes.
struct RebuildArgs {
    const float *p;
    int cap;
    const int32_t *m_dev;
    float nle;
    float4 *kfwd, *kbwd;
    const float4 *slo, *shi;
    int nsx, nsy, nsz, nsuper, ncoarse;
    uint32_t *list, *cnt, *clist, *ccnt;
    int scap;
    int two_level;
    int32_t *status;
    long long *needed;
    int level1_blocks;                 // blocks this field uses in the first launch
    const uint8_t *item_class;         // heavy-first order of the forward's items
    uint32_t *class_hist;
    const uint4 *item_rec;
    uint4 *order_rec;
    int64_t nitems;
};

// Field blockIdx.y: the item order for the next forward (two launches).
__global__ void __launch_bounds__(kOrderChunk) k_class_count_batch(const RebuildArgs *ra) {
    const RebuildArgs &r = ra[blockIdx.y];
    if ((int64_t)blockIdx.x * kOrderChunk >= r.nitems) return;
    class_count_body(r.item_class, r.nitems, r.class_hist, blockIdx.x);
}

// The batch's table of its order over all fields' items (see FwdBatch): pos,
// then place.  One block; a thread per (class, field) sums the chunks' counts.
__device__ __forceinline__ void order_table_body(const RebuildArgs *ra, int nfields, uint32_t *table) {
    __shared__ uint32_t tmp[33];
    const int n = kCostClasses * nfields;
    uint32_t *pos = table, *place = table + n + 1;
    uint32_t carry = 0;
    for (int e0 = 0; e0 < n; e0 += blockDim.x) {
        const int e = e0 + threadIdx.x, f = e % nfields, c = kCostClasses - 1 - e / nfields;
        uint32_t count = 0, heavier = 0;
        if (e < n) {
            const RebuildArgs &r = ra[f];
            const int64_t chunks = (r.nitems + kOrderChunk - 1) / kOrderChunk;
            for (int64_t q = 0; q < chunks; ++q) {
                count += r.class_hist[q * kCostClasses + c];
                for (int h = c + 1; h < kCostClasses; ++h) heavier += r.class_hist[q * kCostClasses + h];
            }
        }
        uint32_t total;
        const uint32_t o = block_exscan(count, tmp, &total);
        if (e < n) {
            pos[e] = carry + o;
            place[e] = heavier;
        }
        carry += total;
    }
    if (threadIdx.x == 0) pos[n] = carry;
}

// The row of blocks past the longest field's chunks makes the table.
__global__ void __launch_bounds__(kOrderChunk) k_order_items_batch(const RebuildArgs *ra, int nfields, uint32_t *table) {
    if (blockIdx.x == gridDim.x - 1) {
        if (blockIdx.y == 0) order_table_body(ra, nfields, table);
        return;
    }
    const RebuildArgs &r = ra[blockIdx.y];
    if ((int64_t)blockIdx.x * kOrderChunk >= r.nitems) return;
    order_items_body(r.item_class, r.class_hist, r.item_rec, r.order_rec, r.nitems, blockIdx.x);
}

// First rebuild launch: one-level fields rebuild, two-level fields list the
// kernels of their blocks of 2 x 2 x 2 super cells; both write the records.
__global__ void __launch_bounds__(kListThreads) k_rebuild_batch(const RebuildArgs *ra) {
    pdl_wait();
    pdl_trigger();
    const RebuildArgs &r = ra[blockIdx.y];
    if ((int)blockIdx.x >= r.level1_blocks) return;
    if (r.two_level)
        coarse_lists_body(r.p, r.cap, r.m_dev, r.nle, r.kfwd, r.kbwd, r.slo, r.shi, r.nsx, r.nsy, r.nsz, r.ncoarse,
                          r.clist, r.ccnt, r.scap, blockIdx.x, r.level1_blocks, 2);
    else
        rebuild_body(r.p, r.cap, r.m_dev, r.nle, r.kfwd, r.kbwd, r.slo, r.shi, r.nsuper, r.list, r.cnt, r.scap,
                     r.status, r.needed, blockIdx.x, r.level1_blocks);
}

// Second rebuild launch: the super-cell lists of two-level fields.
__global__ void __launch_bounds__(kListThreads) k_fine_lists_batch(const RebuildArgs *ra) {
    pdl_wait();
    pdl_trigger();
    const RebuildArgs &r = ra[blockIdx.y];
    if (!r.two_level || (int)blockIdx.x >= r.ncoarse) return;
    child_lists_body<true>(ChildArgs{r.m_dev, r.kfwd, r.slo, r.shi, r.nsx, r.nsy, r.nsz, r.clist, r.ccnt, r.list, r.cnt,
                                     r.scap, r.status, r.needed},
                           blockIdx.x);
}

// ---------------------------------------------------------------- point-major CSR
// One warp per tile; lanes are points.  The super cell's list is walked in
// ascending kernel order, 32 candidates filtered against the tile box at a
// time (one per lane), the kernels that reach it handed round by shuffles, so
// each row comes out sorted.
template <bool FILL>
__global__ void __launch_bounds__(256) k_pmajor(const float *x, const float *y, const float *z, const uint32_t *tile_super,
                                                const uint32_t *tile_start, const float4 *tlo, const float4 *thi,
                                                const uint32_t *cell_start, int cps, int64_t ntiles,
                                                const uint32_t *slist, const uint32_t *scnt, int scap,
                                                const float4 *kfwd, int64_t *rowptr, uint32_t *col) {
    pdl_wait();
    pdl_trigger();
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (t >= ntiles) return;
    const uint32_t s = tile_super[t], p0 = tile_start[t], pe = cell_start[(int64_t)(s + 1) * cps];
    const int64_t i = (int64_t)p0 + lane;
    const bool valid = i < (int64_t)pe;
    const float px = valid ? x[i] : __int_as_float(0x7fc00000);
    const float py = valid ? y[i] : 0.f, pz = valid ? z[i] : 0.f;
    const float4 lo = tlo[t], hi = thi[t];
    const int L = min((int)scnt[s], scap);
    const uint32_t *lst = slist + (size_t)s * scap;
    // a row's entries are written in aligned groups of four: single stores to
    // 32 rows at once took a pass of the store unit each
    uint32_t *row = FILL && valid ? col + rowptr[i] : nullptr;
    const uint32_t phase = (uint32_t)(reinterpret_cast<uintptr_t>(row) >> 2) & 3u;
    uint32_t e0 = 0, e1 = 0, e2 = 0;  // the last three entries
    uint32_t n = 0;
    for (int b = 0; b < L; b += 32) {
        const bool live = b + lane < L;
        const uint32_t j = live ? lst[b + lane] : 0u;
        const float4 k = live ? kfwd[3 * (size_t)j] : make_float4(0.f, 0.f, 0.f, -1.f);
        unsigned hits = __ballot_sync(0xffffffffu, live && box_d2(k.x, k.y, k.z, lo, hi) < k.w);
        while (hits) {
            const int q = __ffs(hits) - 1;
            hits &= hits - 1;
            const float cx = __shfl_sync(0xffffffffu, k.x, q), cy = __shfl_sync(0xffffffffu, k.y, q);
            const float cz = __shfl_sync(0xffffffffu, k.z, q), r2 = __shfl_sync(0xffffffffu, k.w, q);
            const uint32_t jq = __shfl_sync(0xffffffffu, j, q);
            if (in_support(px, py, pz, cx, cy, cz, r2)) {
                if (FILL && ((n + phase) & 3u) == 3u) {
                    if (n >= 3u) {
                        *reinterpret_cast<uint4 *>(row + n - 3) = make_uint4(e0, e1, e2, jq);
                    } else {  // the row begins inside the group
                        row[n] = jq;
                        if (n > 0) row[n - 1] = e2;
                        if (n > 1) row[n - 2] = e1;
                    }
                }
                e0 = e1;
                e1 = e2;
                e2 = jq;
                ++n;
            }
        }
    }
    if (FILL) {  // what the last group lacks
        const uint32_t rest = min(n, (n + phase) & 3u);
        if (rest > 0) row[n - 1] = e2;
        if (rest > 1) row[n - 2] = e1;
        if (rest > 2) row[n - 3] = e0;
    }
    if (!FILL && valid) rowptr[i] = n;
}

// ---------------------------------------------------------------- kernel-major CSR
// kRowParts warps per kernel, each with an equal share of the super cells of
// the support box.  Super cells are visited in ascending id, their tiles in
// ascending order and each tile's points in order, which is ascending binned
// index, so each CSR row comes out sorted: the shares' counts (part) give
// every warp its place in the row.  One warp per kernel took 1.6 ms for 512
// kernels on 64^3 (three warps per SM).
constexpr int kRowParts = 32;
static_assert(kRowParts == 32 && kRowParts + 4 <= kBwdWarpsPerKernel * 22, "a lane per share; the shares' counts fit the standalone adjoint's moments");

template <bool FILL>
__global__ void __launch_bounds__(256, 4) k_kmajor(const float *x, const float *y, const float *z, const float4 *kfwd,
                                                const int32_t *m_dev, serbf_grid g, int sf, int nsx, int nsy,
                                                const float4 *slo, const float4 *shi, const uint32_t *stile0,
                                                const uint32_t *tile_start, const float4 *tlo, const float4 *thi,
                                                const uint32_t *cell_start, int cps, uint32_t *part,
                                                const int64_t *rowptr, uint32_t *col) {
    pdl_wait();
    pdl_trigger();
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, j = (int)(w / kRowParts), share = (int)(w % kRowParts);
    if (j >= *m_dev) return;
    const float4 k = kfwd[3 * (size_t)j];
    const KBox b = kernel_box(k.x, k.y, k.z, k.w, g);
    const int sx0 = b.kx0 / sf, sy0 = b.ky0 / sf, sz0 = b.kz0 / sf;
    const int nx = b.kx1 / sf - sx0 + 1, ny = b.ky1 / sf - sy0 + 1, nz = b.kz1 / sf - sz0 + 1;
    const int64_t all = (int64_t)nx * ny * nz;
    const int64_t q0 = all * share / kRowParts, q1 = all * (share + 1) / kRowParts;
    uint32_t *out = FILL ? col + rowptr[j] + part[w] : nullptr;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t count = 0;
    // 32 super cells at a time, one per lane, then 32 tiles of a reached one
    for (int64_t qb = q0; qb < q1; qb += 32) {
        const int64_t q = qb + lane;
        uint32_t t0 = 0, t1 = 0, pe = 0;
        if (q < q1) {
            const int s = (int)(((sz0 + q / ((int64_t)nx * ny)) * nsy + sy0 + (q / nx) % ny) * nsx + sx0 + q % nx);
            if (box_d2(k.x, k.y, k.z, slo[s], shi[s]) < k.w) {
                t0 = stile0[s];
                t1 = stile0[s + 1];
                pe = cell_start[(int64_t)(s + 1) * cps];
            }
        }
        unsigned sup = __ballot_sync(0xffffffffu, t1 > t0);
        while (sup) {
            const int src = __ffs(sup) - 1;
            sup &= sup - 1;
            const uint32_t a0 = __shfl_sync(0xffffffffu, t0, src), a1 = __shfl_sync(0xffffffffu, t1, src);
            const uint32_t end = __shfl_sync(0xffffffffu, pe, src);
            for (uint32_t tb = a0; tb < a1; tb += 32) {
                const uint32_t t = tb + lane;
                uint32_t start = 0;
                bool hit = false;
                if (t < a1) {
                    hit = box_d2(k.x, k.y, k.z, tlo[t], thi[t]) < k.w;
                    start = tile_start[t];
                }
                unsigned bal = __ballot_sync(0xffffffffu, hit);
                while (bal) {
                    // two tiles at a time: their loads overlap
                    const int ta = __ffs(bal) - 1;
                    bal &= bal - 1;
                    const int tz = bal ? __ffs(bal) - 1 : ta;
                    const bool two = bal != 0;
                    bal &= bal - 1;
                    const uint32_t i = __shfl_sync(0xffffffffu, start, ta) + lane, i2 = __shfl_sync(0xffffffffu, start, tz) + lane;
                    const bool v = i < end, v2 = two && i2 < end;
                    const float xa = v ? x[i] : 0.f, ya = v ? y[i] : 0.f, za = v ? z[i] : 0.f;
                    const float xb = v2 ? x[i2] : 0.f, yb = v2 ? y[i2] : 0.f, zb = v2 ? z[i2] : 0.f;
                    const bool in = v && in_support(xa, ya, za, k.x, k.y, k.z, k.w);
                    const bool in2 = v2 && in_support(xb, yb, zb, k.x, k.y, k.z, k.w);
                    const unsigned m = __ballot_sync(0xffffffffu, in), m2 = __ballot_sync(0xffffffffu, in2);
                    if (FILL && in) out[count + __popc(m & lt)] = i;
                    count += __popc(m);
                    if (FILL && in2) out[count + __popc(m2 & lt)] = i2;
                    count += __popc(m2);
                }
            }
        }
    }
    if (!FILL && lane == 0) part[w] = count;
}

// A warp per kernel: its shares' counts become places in the row, its total
// goes to rowptr[j].
__global__ void __launch_bounds__(256) k_row_parts(const int32_t *m_dev, uint32_t *part, int64_t *rowptr) {
    pdl_wait();
    pdl_trigger();
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (j >= *m_dev) return;
    const uint32_t v = part[(size_t)j * kRowParts + lane], inc = warp_iscan(v);
    part[(size_t)j * kRowParts + lane] = inc - v;
    if (lane == 31) rowptr[j] = inc;
}

bool ws_ok(const serbf_workspace *ws) { return ws && ws->magic == kMagic && ws->binned; }

// Two levels when asked, or by default once super cells x kernel capacity
// reaches 2^25 box tests: measured, the 256^3 band workload (4913 super
// cells, capacity 32768) rebuilds 4x faster in two levels, while the 128^3
// one (729, 8192) is slower by the extra launch.
bool rebuild_two_level(int levels, int64_t nsuper, int cap) {
    return levels >= 2 || (levels == 0 && nsuper * (int64_t)cap >= (int64_t)1 << 25);
}

// Three levels (blocks of 4 x 4 x 4 super cells against every kernel, then
// blocks of 2 x 2 x 2, then super cells) when asked, or by default once the
// second level alone would make 2^25 box tests: measured, the 256^3 band
// with super cells of 2 x 2 x 2 cells (4913 blocks of 2 x 2 x 2, capacity
// 32768) rebuilds in a fraction of its two-level time.  Single fields only;
// the batched epoch takes two levels.
bool rebuild_three_level(int levels, int64_t ncoarse, int cap) {
    return levels == 3 || (levels == 0 && ncoarse * (int64_t)cap >= (int64_t)1 << 25);
}

}  // namespace

namespace serbf {

size_t rebuild_args_size() { return sizeof(RebuildArgs); }

// Host record of one field's neighbour rebuild for a batch (out:
// sizeof(RebuildArgs) bytes); *level1_blocks, *chunks and *parents (blocks of
// super cells of a field that takes two levels, else 0) size the batch's grids.
int batch_rebuild_args(const serbf_points *pts, const serbf_params *prm, const serbf_config *cfg,
                       serbf_workspace *ws, int warps, void *out, int *level1_blocks, int64_t *chunks, int *parents) {
    if (!pts || !prm || !cfg || !ws_ok(ws)) return SERBF_EINVAL;
    if (!prm->p || !prm->m || prm->cap < 1 || prm->cap > ws->sz.max_kernels) return SERBF_EINVAL;
    if (pts->n != ws->npoints) return SERBF_EINVAL;
    if (!(cfg->eps > 0.0 && cfg->eps < 1.0) || cfg->rebuild_levels < 0 || cfg->rebuild_levels > 3) return SERBF_EINVAL;
    RebuildArgs r;
    memset(&r, 0, sizeof(r));
    const int nsx = ws->ns[0], nsy = ws->ns[1], nsz = ws->ns[2];
    const int64_t ncoarse = (int64_t)((nsx + 1) / 2) * ((nsy + 1) / 2) * ((nsz + 1) / 2);
    const int prep_blocks = (prm->cap + 255) / 256;
    r.p = prm->p;
    r.cap = prm->cap;
    r.m_dev = prm->m;
    r.nle = (float)(-log(cfg->eps));
    r.kfwd = ws->kfwd;
    r.kbwd = ws->kbwd;
    r.slo = ws->sup_lo;
    r.shi = ws->sup_hi;
    r.nsx = nsx;
    r.nsy = nsy;
    r.nsz = nsz;
    r.nsuper = ws->nsuper;
    r.ncoarse = (int)ncoarse;
    r.list = ws->sup_list;
    r.cnt = ws->sup_cnt;
    r.clist = ws->crs_list;
    r.ccnt = ws->crs_cnt;
    r.scap = ws->sz.super_cap;
    r.two_level = rebuild_two_level(cfg->rebuild_levels, ws->nsuper, prm->cap) && ncoarse <= ws->max_coarse;
    r.status = ws->status;
    r.needed = ws->needed;
    r.level1_blocks = (r.two_level ? (int)ncoarse : ws->nsuper) + prep_blocks;
    const ItemSet &items = items_of(ws, warps);
    r.item_class = items.cls;
    r.class_hist = ws->class_hist;
    r.item_rec = items.rec;
    r.order_rec = items.order;
    r.nitems = items.n;
    memcpy(out, &r, sizeof(r));
    *level1_blocks = r.level1_blocks;
    *chunks = (items.n + kOrderChunk - 1) / kOrderChunk;
    *parents = r.two_level ? r.ncoarse : 0;
    return SERBF_OK;
}

// The batched rebuild: item order (two launches), then the lists and
// records (one launch, two when some field takes two levels).
int batch_rebuild_launch(const void *args, int nfields, int level1_blocks, int64_t chunks, int parents, uint32_t *table,
                         cudaStream_t s) {
    const RebuildArgs *ra = static_cast<const RebuildArgs *>(args);
    if (chunks > 0) {
        k_class_count_batch<<<dim3((unsigned)chunks, (unsigned)nfields), kOrderChunk, 0, s>>>(ra);
        k_order_items_batch<<<dim3((unsigned)chunks + 1, (unsigned)nfields), kOrderChunk, 0, s>>>(ra, nfields, table);
    }
    launch_pdl(k_rebuild_batch, dim3((unsigned)level1_blocks, (unsigned)nfields), dim3(kListThreads), 0, s, ra);
    if (parents) launch_pdl(k_fine_lists_batch, dim3((unsigned)parents, (unsigned)nfields), dim3(kListThreads), 0, s, ra);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

}  // namespace serbf

extern "C" int serbf_build_neighbors(const serbf_points *pts, const serbf_params *prm, const serbf_config *cfg,
                                     serbf_csr *kmajor, serbf_csr *pmajor, int64_t *npairs, serbf_workspace *ws,
                                     void *stream) {
    SERBF_TRACE();
    if (!pts || !prm || !cfg || !ws_ok(ws)) return SERBF_EINVAL;
    if (!prm->p || !prm->m || prm->cap < 1 || prm->cap > ws->sz.max_kernels) return SERBF_EINVAL;
    if (pts->n != ws->npoints || (pts->n > 0 && (!pts->x || !pts->y || !pts->z))) return SERBF_EINVAL;
    if (!(cfg->eps > 0.0 && cfg->eps < 1.0)) return SERBF_EINVAL;
    if (cfg->rebuild_levels < 0 || cfg->rebuild_levels > 3) return SERBF_EINVAL;
    if (kmajor && (!kmajor->rowptr || (kmajor->cap > 0 && !kmajor->col))) return SERBF_EINVAL;
    if (pmajor && (!pmajor->rowptr || (pmajor->cap > 0 && !pmajor->col))) return SERBF_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    // fork: the item order for the next forward overlaps the rebuild.  Nothing
    // to order when no forward has measured since the binning, whose order is
    // there already -- except under capture, where the graph will be replayed
    // after forwards that do measure.
    const ItemSet &items = items_of(ws, forward_warps(ws->items[1].n, ws->sm_count, cfg->fwd_warps));
    bool measured = !ws->unmeasured;
    if (!measured) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {
            cudaGetLastError();  // another stream's capture forbids the question on the default stream
            measured = true;
        }
        measured |= capture != cudaStreamCaptureStatusNone;
    }
    const bool fork = items.n > 0 && ws->aux && measured;
    if (fork) {
        if (cudaEventRecord(ws->ev_fork, s) != cudaSuccess) return SERBF_ECUDA;
        if (cudaStreamWaitEvent(ws->aux, ws->ev_fork, 0) != cudaSuccess) return SERBF_ECUDA;
        const unsigned nchunks = (unsigned)((items.n + kOrderChunk - 1) / kOrderChunk);
        // few items: every block counts all classes itself, one launch less on
        // the way to the forward
        const bool direct = order_direct(ws->npoints, ws->nsuper);
        if (!direct) k_class_count<<<nchunks, kOrderChunk, 0, ws->aux>>>(items.cls, items.n, ws->class_hist);
        k_order_items<<<nchunks, kOrderChunk, 0, ws->aux>>>(items.cls, direct ? nullptr : ws->class_hist, items.rec,
                                                            items.order, items.n);
        SERBF_CHECK_LAUNCH();
        if (cudaEventRecord(ws->ev_join, ws->aux) != cudaSuccess) return SERBF_ECUDA;
    }
    {
        const float nle = (float)(-log(cfg->eps));
        const int prep_blocks = (prm->cap + 255) / 256;
        const int nsx = ws->ns[0], nsy = ws->ns[1], nsz = ws->ns[2];
        const int64_t ncoarse = (int64_t)((nsx + 1) / 2) * ((nsy + 1) / 2) * ((nsz + 1) / 2);
        const int64_t ntop = (int64_t)((nsx + 3) / 4) * ((nsy + 3) / 4) * ((nsz + 3) / 4);
        if (rebuild_two_level(cfg->rebuild_levels, ws->nsuper, prm->cap) && ncoarse <= ws->max_coarse) {
            if (rebuild_three_level(cfg->rebuild_levels, ncoarse, prm->cap) && ntop <= ws->nsuper) {
                // blocks of 4 x 4 x 4 super cells against every kernel (their
                // lists and counts held in the super cells' storage, which the
                // last level rewrites), then blocks of 2 x 2 x 2
                launch_pdl(k_coarse_lists, dim3((unsigned)(ntop + prep_blocks)), dim3(kListThreads), 0, s,
                           (const float *)prm->p, prm->cap, (const int32_t *)prm->m, nle, ws->kfwd, ws->kbwd,
                           (const float4 *)ws->sup_lo, (const float4 *)ws->sup_hi, nsx, nsy, nsz, (int)ntop,
                           ws->sup_list, ws->sup_cnt, ws->sz.super_cap, 4);
                launch_pdl(k_child_lists<false>, dim3((unsigned)ntop), dim3(kListThreads), 0, s,
                           ChildArgs{prm->m, ws->kfwd, ws->sup_lo, ws->sup_hi, nsx, nsy, nsz, ws->sup_list, ws->sup_cnt,
                                     ws->crs_list, ws->crs_cnt, ws->sz.super_cap, ws->status, ws->needed});
            } else {
                launch_pdl(k_coarse_lists, dim3((unsigned)(ncoarse + prep_blocks)), dim3(kListThreads), 0, s,
                           (const float *)prm->p, prm->cap, (const int32_t *)prm->m, nle, ws->kfwd, ws->kbwd,
                           (const float4 *)ws->sup_lo, (const float4 *)ws->sup_hi, nsx, nsy, nsz, (int)ncoarse,
                           ws->crs_list, ws->crs_cnt, ws->sz.super_cap, 2);
            }
            launch_pdl(k_child_lists<true>, dim3((unsigned)ncoarse), dim3(kListThreads), 0, s,
                       ChildArgs{prm->m, ws->kfwd, ws->sup_lo, ws->sup_hi, nsx, nsy, nsz, ws->crs_list, ws->crs_cnt,
                                 ws->sup_list, ws->sup_cnt, ws->sz.super_cap, ws->status, ws->needed});
        } else {
            launch_pdl(k_rebuild, dim3(ws->nsuper + prep_blocks), dim3(kListThreads), 0, s, (const float *)prm->p, prm->cap,
                       (const int32_t *)prm->m, nle, ws->kfwd, ws->kbwd, (const float4 *)ws->sup_lo,
                       (const float4 *)ws->sup_hi, ws->nsuper, ws->sup_list, ws->sup_cnt, ws->sz.super_cap,
                       ws->status, ws->needed);
        }
    }
    int rc = SERBF_OK;
    SERBF_CHECK_LAUNCH();
    // join the side stream
    if (fork && cudaStreamWaitEvent(s, ws->ev_join, 0) != cudaSuccess) return SERBF_ECUDA;
    if (!kmajor && !pmajor) return SERBF_OK;

    // Explicit lists: an overflowing candidate list would make them silently
    // incomplete, so the status is checked first.
    int32_t flags;
    rc = serbf_status(ws, &flags, nullptr, 0, stream);
    if (rc) return rc;
    int32_t m = 0;
    if (cudaMemcpyAsync(&m, prm->m, sizeof(int32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess) return SERBF_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
    const int cps = ws->sf * ws->sf * ws->sf;
    int64_t n = pts->n;
    int64_t total = -1;
    int result = SERBF_OK;
    // scratch of the explicit lists, idle outside the standalone adjoint
    uint32_t *part = reinterpret_cast<uint32_t *>(ws->moments);
    if (kmajor) {
        const unsigned blocks = (unsigned)(((int64_t)m * kRowParts * 32 + 255) / 256);
        if (m > 0) {
            launch_pdl(k_kmajor<false>, dim3(blocks), dim3(256), 0, s, pts->x, pts->y, pts->z, ws->kfwd, prm->m, ws->grid,
                       ws->sf, ws->ns[0], ws->ns[1], ws->sup_lo, ws->sup_hi, ws->super_tile0, ws->tile_start, ws->tile_lo,
                       ws->tile_hi, ws->cell_start, cps, part, kmajor->rowptr, nullptr);
            launch_pdl(k_row_parts, dim3((unsigned)((m + 7) / 8)), dim3(256), 0, s, prm->m, part, kmajor->rowptr);
        }
        rc = launch_exscan_i64(kmajor->rowptr, m, reinterpret_cast<int64_t *>(part + (size_t)m * kRowParts), s);
        if (rc) return rc;
        int64_t tot = 0;
        if (cudaMemcpyAsync(&tot, kmajor->rowptr + m, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess)
            return SERBF_ECUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
        total = tot;
        if (tot > kmajor->cap) result = SERBF_ECAPACITY;
        else if (m > 0)
            launch_pdl(k_kmajor<true>, dim3(blocks), dim3(256), 0, s, pts->x, pts->y, pts->z, ws->kfwd, prm->m, ws->grid,
                       ws->sf, ws->ns[0], ws->ns[1], ws->sup_lo, ws->sup_hi, ws->super_tile0, ws->tile_start, ws->tile_lo,
                       ws->tile_hi, ws->cell_start, cps, part, kmajor->rowptr, kmajor->col);
        SERBF_CHECK_LAUNCH();
    }
    if (pmajor) {
        int64_t nt = ws->ntiles;
        const unsigned blocks = (unsigned)((nt * 32 + 255) / 256);
        if (nt > 0)
            launch_pdl(k_pmajor<false>, dim3(blocks), dim3(256), 0, s, pts->x, pts->y, pts->z, ws->tile_super, ws->tile_start,
                                                   ws->tile_lo, ws->tile_hi, ws->cell_start, cps, nt, ws->sup_list,
                                                   ws->sup_cnt, ws->sz.super_cap, ws->kfwd, pmajor->rowptr, nullptr);
        rc = launch_exscan_i64(pmajor->rowptr, n, reinterpret_cast<int64_t *>(ws->nz), s);
        if (rc) return rc;
        int64_t tot = 0;
        if (cudaMemcpyAsync(&tot, pmajor->rowptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess)
            return SERBF_ECUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
        total = tot;
        if (tot > pmajor->cap) result = SERBF_ECAPACITY;
        else if (nt > 0)
            launch_pdl(k_pmajor<true>, dim3(blocks), dim3(256), 0, s, pts->x, pts->y, pts->z, ws->tile_super, ws->tile_start,
                                                  ws->tile_lo, ws->tile_hi, ws->cell_start, cps, nt, ws->sup_list,
                                                  ws->sup_cnt, ws->sz.super_cap, ws->kfwd, pmajor->rowptr,
                                                  pmajor->col);
        SERBF_CHECK_LAUNCH();
    }
    if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
    if (npairs) *npairs = total;
    return result;
}
