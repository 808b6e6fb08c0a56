// Initial kernels: Algorithm 1 (greedy largest inscribed spheres over the
// interior training points) and Eq. 3-12 (isotropic axis parameters from the
// nearest other centre), once before the fit.
//
// The interior points (1 < t < 2, Eq. 3-10) are sorted by d_in = |S|
// descending (stable, so equal values keep the binned order: the first
// maximum is taken, as an argmax does).  The greedy walk of that order is done
// in rounds: one block takes the next kBatch points that are still there and
// settles them among themselves in order (k_settle), then all blocks remove
// the later points that the new centres' spheres cover (k_cover).  That is the
// same walk: a point's fate depends only on earlier centres, all of which are
// known when it is settled.  The removal test is the float squared distance in
// the support predicate's operation order against fl(r r), so the decisions
// are exact and reproducible.
//
// One block walking point by point took 100 ms for 23 k interior points and
// 6457 centres (64^3, 15 us a centre, nearly all of it barriers and dependent
// loads); ten rounds take 0.9 ms, two thirds of it in k_settle's one block.
#include <math.h>

#include "common.cuh"

using namespace serbf;

namespace {

constexpr int kBatch = 1024;      // points settled per round, one per thread
constexpr int kRounds = 8;        // rounds between two looks at the state
// New centres in a round after which the next one looks for conflicts first
// (40^3 / 64^3 / 80^3 points: 410 / 890 / 1107 us, never looking 826 / 2122 / 3150).
constexpr uint32_t kSparse = 384;

// Where the walk stands (device; ws->counters + 8).
struct Walk {
    uint32_t next;     // first sorted position not settled yet
    uint32_t fresh;    // centres of the last round
    uint32_t count;    // interior points
    uint32_t centres;  // centres so far
};

// Sort keys: interior points by |S| descending (inverted float bits of a
// positive value), everything else last.
__global__ void k_init_keys(const float *t, const float *S, int64_t n, uint32_t *keys, uint32_t *vals,
                            uint32_t *count) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const bool in = (1.0f < t[i]) && (t[i] < 2.0f);
        keys[i] = in ? ~__float_as_uint(fabsf(S[i])) : 0xffffffffu;
        vals[i] = (uint32_t)i;
        const unsigned b = __ballot_sync(__activemask(), in);
        if ((threadIdx.x & 31) == __ffs(__activemask()) - 1 && b) atomicAdd(count, (uint32_t)__popc(b));
    }
}

// Interior points in sorted order as (x, y, z, fl(r r)).
__global__ void k_init_points(const float *x, const float *y, const float *z, const float *S, const uint32_t *order,
                              const Walk *w, float4 *pts) {
    const int64_t nin = w->count;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nin; q += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = order[q];
        const float r = fabsf(S[i]);
        pts[q] = make_float4(x[i], y[i], z[i], __fmul_rn(r, r));
    }
}

// Whether the sphere of c (centre, r r) holds p.
__device__ __forceinline__ bool covered(float4 p, float4 c) {
    return !(support_d2(__fsub_rn(p.x, c.x), __fsub_rn(p.y, c.y), __fsub_rn(p.z, c.z)) > c.w);
}

static_assert(kBatch * 16 <= 256 * (kDirectBlocks + 1) * 4, "the fresh centres fit the sort's histograms");

struct WalkArgs {
    Walk *w;
    float4 *pts;            // interior points in order; settled places take the centres
    const uint32_t *order;  // binned indices of the interior points, |S| descending
    uint8_t *removed;       // per sorted position
    uint32_t *centres;      // binned indices of the centres, in selection order
    float4 *fresh;          // the last round's centres
    int32_t cap;
};

// One block: the next kBatch points still there, settled in order.  Thread c
// holds the c-th of them.  Each step takes the first one left that may cover
// another and lets every later thread test its point, one barrier a step.
// After a round with many centres the spheres are small and most points cover
// none of the batch, so all pairs are tested first and only the points that do
// cover a later one are stepped through.
__global__ void __launch_bounds__(kBatch) k_settle(WalkArgs a) {
    pdl_wait();
    pdl_trigger();
    __shared__ float4 s_pt[kBatch];
    __shared__ uint32_t s_pos[kBatch];
    __shared__ uint32_t s_word[2][kBatch / 32];
    __shared__ uint8_t s_covers[kBatch];
    __shared__ uint32_t tmp[33];
    __shared__ uint32_t s_next;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t nin = a.w->count, first = a.w->next, last = a.w->fresh, before = a.w->centres;
    if (first >= nin) {
        if (tid == 0) a.w->fresh = 0u;
        return;
    }
    if (tid == 0) s_next = nin;
    __syncthreads();
    uint32_t n = 0;
    for (uint64_t b = first; b < nin && n < kBatch; b += 4 * kBatch) {
        const uint64_t q0 = b + 4 * tid;
        uint32_t here = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) here |= (q0 + k < nin && !a.removed[q0 + k] ? 1u : 0u) << k;
        uint32_t tot, o = block_exscan(__popc(here), tmp, &tot) + n;
        for (; here && o < kBatch; here &= here - 1, ++o) {
            const uint32_t q = (uint32_t)q0 + __ffs(here) - 1;
            s_pos[o] = q;
            if (o == kBatch - 1) s_next = q + 1;
        }
        n += tot;
    }
    n = min(n, (uint32_t)kBatch);
    __syncthreads();
    const bool mine = tid < (int)n;
    const float4 p = mine ? a.pts[s_pos[tid]] : make_float4(0.f, 0.f, 0.f, 0.f);
    s_pt[tid] = p;
    const bool sparse = last >= kSparse;
    s_covers[tid] = !sparse;
    __syncthreads();
    if (sparse) {
        if (mine)
            for (int i = 0; i < tid; ++i)
                if (covered(p, s_pt[i])) s_covers[i] = 1;
        __syncthreads();
    }
    const bool covers = s_covers[tid];
    bool left = mine;
    for (int cur = -1, buf = 0;; buf ^= 1) {
        const unsigned bal = __ballot_sync(0xffffffffu, left && covers && tid > cur);
        if (lane == 0) s_word[buf][warp] = bal;
        __syncthreads();
        const uint32_t word = s_word[buf][lane];
        const unsigned some = __ballot_sync(0xffffffffu, word != 0u);
        if (!some) break;
        const int w = __ffs(some) - 1;
        cur = 32 * w + __ffs(__shfl_sync(0xffffffffu, word, w)) - 1;
        if (left && tid > cur && covered(p, s_pt[cur])) left = false;
    }
    uint32_t tot;
    const uint32_t o = block_exscan(left, tmp, &tot);
    if (left) {
        if (before + o < (uint32_t)a.cap) a.centres[before + o] = a.order[s_pos[tid]];
        a.fresh[o] = p;
        a.pts[before + o] = p;  // at or before this point's own place, which is settled
    }
    if (tid == 0) {
        a.w->next = s_next;
        a.w->fresh = tot;
        a.w->centres = before + tot;
    }
}

// The points from the next position on that a new centre covers are removed:
// blocks (x, y) test their points against the y-th kCoverPart of the new
// centres (all of them by one thread were a chain of up to 1024 tests, 26 us
// a round).
constexpr int kCoverPart = 128;
__global__ void __launch_bounds__(256) k_cover(WalkArgs a) {
    pdl_wait();
    pdl_trigger();
    __shared__ float4 c[kCoverPart];
    const uint32_t nin = a.w->count, fresh = a.w->fresh, next = a.w->next, first = blockIdx.y * kCoverPart;
    if (first >= fresh) return;
    const int k = (int)min((uint32_t)kCoverPart, fresh - first);
    if (threadIdx.x < k) c[threadIdx.x] = a.fresh[first + threadIdx.x];
    __syncthreads();
    for (uint64_t q0 = (uint64_t)next + blockIdx.x * 256ull; q0 < nin; q0 += gridDim.x * 256ull) {
        const uint64_t q = q0 + threadIdx.x;
        bool here = q < nin && !a.removed[q];
        const float4 p = here ? a.pts[q] : make_float4(0.f, 0.f, 0.f, 0.f);
        bool gone = false;
        if (here)
            for (int i = 0; i < k && !gone; ++i) gone = covered(p, c[i]);
        if (gone) a.removed[q] = 1;
    }
}

// Eq. 3-12 for the selected centres (a warp per kNearest centres, which share
// the coordinates that it reads): dhat = distance to
// the nearest other centre (a single centre: twice its radius), then
// d = 2 sqrt(-ln(gamma / w^2)) / dhat on all axes, angles 0, w = t.
constexpr int kNearest = 4;
__global__ void k_init_params(const float *x, const float *y, const float *z, const float *t, const float *S,
                              const uint32_t *centres, const float4 *at, const uint32_t *ncentres, int32_t cap,
                              float gamma, float *p, int32_t *m_dev) {
    const int M = (int)min(*ncentres, (uint32_t)cap);
    const int j0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kNearest, lane = threadIdx.x & 31;
    if (j0 == 0 && lane == 0) *m_dev = M;
    if (j0 >= M) return;
    float4 c[kNearest];
    float near[kNearest];
#pragma unroll
    for (int k = 0; k < kNearest; ++k) {
        c[k] = at[min(j0 + k, M - 1)];
        near[k] = INFINITY;
    }
    for (int i = lane; i < M; i += 32) {
        const float4 q = at[i];
#pragma unroll
        for (int k = 0; k < kNearest; ++k) {
            const float dx = q.x - c[k].x, dy = q.y - c[k].y, dz = q.z - c[k].z;
            const float d2 = dx * dx + dy * dy + dz * dz;
            if (i != j0 + k) near[k] = fminf(near[k], d2);
        }
    }
#pragma unroll
    for (int k = 0; k < kNearest; ++k) near[k] = -warp_max(-near[k]);
    const int j = j0 + lane;
    if (lane >= kNearest || j >= M) return;
    float best = near[0];
#pragma unroll
    for (int k = 1; k < kNearest; ++k) best = lane == k ? near[k] : best;
    const uint32_t cj = centres[j];
    const float px = x[cj], py = y[cj], pz = z[cj];
    const float dhat = M > 1 ? sqrtf(best) : 2.f * fabsf(S[cj]);
    const float w = t[cj];
    const float d = 2.f * sqrtf(-logf(gamma / (w * w))) / dhat;
    p[PCX * cap + j] = px;
    p[PCY * cap + j] = py;
    p[PCZ * cap + j] = pz;
    p[PD1 * cap + j] = d;
    p[PD2 * cap + j] = d;
    p[PD3 * cap + j] = d;
    p[PTX * cap + j] = 0.f;
    p[PTY * cap + j] = 0.f;
    p[PTZ * cap + j] = 0.f;
    p[PW * cap + j] = w;
}

}  // namespace

extern "C" int serbf_init_kernels(const serbf_points *pts, const float *S_raw, double gamma, serbf_params *prm,
                                  int32_t *m_out, serbf_workspace *ws, void *stream) {
    SERBF_TRACE();
    if (!pts || !prm || !prm->p || !prm->m || prm->cap < 1 || !ws || ws->magic != kMagic || !ws->binned)
        return SERBF_EINVAL;
    if (pts->n != ws->npoints || prm->cap > ws->sz.max_kernels || !(gamma > 0.0 && gamma < 1.0)) return SERBF_EINVAL;
    const int64_t n = pts->n;
    if (n > 0 && (!pts->x || !pts->y || !pts->z || !pts->t || !S_raw)) return SERBF_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    Walk *w = reinterpret_cast<Walk *>(ws->counters + 8);
    if (cudaMemsetAsync(w, 0, sizeof(Walk), s) != cudaSuccess) return SERBF_ECUDA;
    uint32_t *k = ws->keys0, *v = ws->vals0, *kt = ws->keys1, *vt = ws->vals1;
    const int grid = (int)((n + 255) / 256 < 152 * 64 ? (n + 255) / 256 : 152 * 64);
    uint32_t found = 0;
    if (n > 0) {
        k_init_keys<<<grid, 256, 0, s>>>(pts->t, S_raw, n, k, v, &w->count);
        int rc = radix_sort_pairs(&k, &v, &kt, &vt, n, 32, ws->hist, s);
        if (rc) return rc;
        // kt now holds the removal flags, the sort's other value buffer the
        // centres, its histograms the last round's centres; the points lie in
        // the adjoint's compaction buffer (16 bytes per point, idle here)
        WalkArgs a{w, ws->nz, v, reinterpret_cast<uint8_t *>(kt), vt, reinterpret_cast<float4 *>(ws->hist), prm->cap};
        k_init_points<<<grid, 256, 0, s>>>(pts->x, pts->y, pts->z, S_raw, v, w, ws->nz);
        if (cudaMemsetAsync(kt, 0, (size_t)n, s) != cudaSuccess) return SERBF_ECUDA;
        const int64_t cover = (n + 255) / 256, most = 8 * (int64_t)ws->sm_count;
        Walk now;
        do {
            // ends: every round settles at least one point
            for (int q = 0; q < kRounds; ++q) {
                launch_pdl(k_settle, dim3(1), dim3(kBatch), 0, s, a);
                launch_pdl(k_cover, dim3((unsigned)(cover < most ? cover : most), kBatch / kCoverPart), dim3(256), 0, s, a);
            }
            SERBF_CHECK_LAUNCH();
            if (cudaMemcpyAsync(&now, w, sizeof(Walk), cudaMemcpyDeviceToHost, s) != cudaSuccess) return SERBF_ECUDA;
            if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
        } while (now.next < now.count);
        found = now.centres;
        k_init_params<<<(unsigned)((prm->cap + 8 * kNearest - 1) / (8 * kNearest)), 256, 0, s>>>(
            pts->x, pts->y, pts->z, pts->t, S_raw, vt, ws->nz, &w->centres, prm->cap, (float)gamma, prm->p, prm->m);
    } else {
        if (cudaMemsetAsync(prm->m, 0, sizeof(int32_t), s) != cudaSuccess) return SERBF_ECUDA;
    }
    SERBF_CHECK_LAUNCH();
    if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
    if (m_out) *m_out = (int32_t)found;
    return (int64_t)found > prm->cap ? SERBF_ECAPACITY : SERBF_OK;
}
