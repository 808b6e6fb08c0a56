// Workspace management, configuration, status, Eq. 3-10 normalisation and
// small utility kernels (scans, gathers).
#include <math.h>
#include <string.h>

#include "common.cuh"

using namespace serbf;

namespace {

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

int64_t max_supers_for(int64_t cells, int sf) {
    double e = cbrt((double)cells);
    int64_t per = (int64_t)ceil(e / sf) + 1;
    int64_t s = per * per * per;
    return s < 1 ? 1 : s;
}

// Walks the carve-up; with base == nullptr it only sizes.
struct Carver {
    char *base;
    size_t off = 0;
    template <typename T>
    T *take(int64_t count) {
        off = align_up(off, 256);
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += sizeof(T) * (size_t)(count > 0 ? count : 1);
        return p;
    }
};

bool sizes_ok(const serbf_ws_sizes *s) {
    return s && s->max_points > 0 && s->max_points < (1ll << 31) && s->max_kernels > 0 && s->max_cells > 0 &&
           s->super_cap > 0 && s->super_factor >= 1 && s->super_factor <= 16;
}

void carve(Carver &c, serbf_workspace *w, const serbf_ws_sizes *s) {
    int64_t N = s->max_points, K = s->max_kernels, C = s->max_cells;
    int64_t S = max_supers_for(C, s->super_factor);
    int64_t cps = (int64_t)s->super_factor * s->super_factor * s->super_factor;
    int64_t T = N / kTile + S + 1;
    int64_t SB = (N + kSortTile - 1) / kSortTile;
    if (SB < 1) SB = 1;
    w->max_tiles = T;
    w->max_supers = S;
    w->sort_blocks = SB;
    w->keys0 = c.take<uint32_t>(N);
    w->keys1 = c.take<uint32_t>(N);
    w->vals0 = c.take<uint32_t>(N);
    w->vals1 = c.take<uint32_t>(N);
    w->hist = c.take<uint32_t>(256 * (SB > kDirectBlocks ? SB : kDirectBlocks) + 256);
    w->cell_start = c.take<uint32_t>(S * cps + 1);
    w->super_tile0 = c.take<uint32_t>(S + 1);
    w->tile_super = c.take<uint32_t>(T);
    w->tile_start = c.take<uint32_t>(T);
    for (int k = 0; k < 2; ++k) {
        ItemSet &it = w->items[k];
        const int64_t I = T / (k ? kMostTiles : 2) + S + 2;
        it.super0 = c.take<uint32_t>(S + 1);
        it.rec = c.take<uint4>(I);
        it.order = c.take<uint4>(I);
        it.cls = c.take<uint8_t>(I);
        it.sched = c.take<uint32_t>(4);
        it.total = c.take<unsigned long long>(2);
    }
    w->class_hist = c.take<uint32_t>((T / 2 + S + 2 + kOrderChunk - 1) / kOrderChunk * kCostClasses);
    w->tile_lo = c.take<float4>(T);
    w->tile_hi = c.take<float4>(T);
    w->sup_lo = c.take<float4>(S);
    w->sup_hi = c.take<float4>(S);
    w->kfwd = c.take<float4>(3 * K);
    w->kbwd = c.take<float4>(4 * K);
    w->sup_list = c.take<uint32_t>(S * (int64_t)s->super_cap);
    w->sup_cnt = c.take<uint32_t>(S);
    // balanced grids have about S / 8 blocks of 2 x 2 x 2 super cells; flat
    // ones more, and those rebuild in one level
    w->max_coarse = S / 4 + 16;
    w->crs_list = c.take<uint32_t>(w->max_coarse * (int64_t)s->super_cap);
    w->crs_cnt = c.take<uint32_t>(w->max_coarse);
    w->fwd_part = c.take<FwdPart>(T + 1);
    w->fwd_gpart = c.take<FwdPart>(T / kFwdGroup + 2);
    w->bwd_pairs = c.take<unsigned long long>(K);
    w->adj_fix = c.take<unsigned long long>(K * 10);
    w->adj_pairs = c.take<unsigned long long>(8);
    w->moments = c.take<float>((int64_t)K * kBwdWarpsPerKernel * 22);
    w->nzrec = c.take<float4>(2 * T);
    w->nzc_cnt = c.take<uint32_t>(T);
    w->nz = c.take<float4>(T * kTile);
    w->step_part = c.take<float>(6 * (SERBF_NPARAM * (K / 256 + 1) + 1));
    w->step_scal = c.take<double>(8);
    w->sel_hist = c.take<uint32_t>(kSelBins);
    w->sel_ctl = c.take<uint32_t>(16);
    w->add_info = c.take<int32_t>(16);
    w->status = c.take<int32_t>(16);
    w->needed = c.take<long long>(4);
    w->counters = c.take<uint32_t>(16);
    w->dtmp = c.take<double>(16);
    w->cell_max = c.take<uint32_t>(4);
    w->field_box = c.take<float4>(2);
}

// Exclusive scan in three launches: sums of tiles of kScanTile elements, a scan
// of those by one block, then every tile with its base.  (One block over all
// elements: 216 us for 262 144.)
constexpr int kScanThreads = 512;
constexpr int kScanPer = 8;

__device__ __forceinline__ int64_t block_iscan_i64(int64_t v, long long *tmp, int64_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) tmp[warp] = inc;
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
    inc += warp ? tmp[warp - 1] : 0ll;
    __syncthreads();
    return inc;
}

// SUMS: the tile's sum to tiles[b]; otherwise the exclusive scan of the tile
// from tiles[b] on (the last tile also writes a[n]).
template <bool SUMS>
__global__ void __launch_bounds__(kScanThreads) k_scan_tile(int64_t *a, int64_t n, int64_t *tiles) {
    pdl_wait();
    pdl_trigger();
    __shared__ long long tmp[32];
    const int64_t base = blockIdx.x * (int64_t)kScanTile;
    int64_t carry = SUMS ? 0 : tiles[blockIdx.x];
    for (int r = 0; r < kScanPer; ++r) {
        const int64_t i = base + r * kScanThreads + threadIdx.x;
        const int64_t v = i < n ? a[i] : 0;
        int64_t total;
        const int64_t inc = block_iscan_i64(v, tmp, &total);
        if (!SUMS && i < n) a[i] = carry + inc - v;
        carry += total;
    }
    if (threadIdx.x == 0) {
        if (SUMS) tiles[blockIdx.x] = carry;
        else if (blockIdx.x == gridDim.x - 1) a[n] = carry;
    }
}

__global__ void __launch_bounds__(1024) k_scan_sums(int64_t *tiles, int64_t nt) {
    pdl_wait();
    pdl_trigger();
    __shared__ long long tmp[32];
    int64_t carry = 0;
    for (int64_t t0 = 0; t0 < nt; t0 += blockDim.x) {
        const int64_t t = t0 + threadIdx.x, v = t < nt ? tiles[t] : 0;
        int64_t total;
        const int64_t inc = block_iscan_i64(v, tmp, &total);
        if (t < nt) tiles[t] = carry + inc - v;
        carry += total;
    }
}

__global__ void k_gather(const float *src, const uint32_t *perm, float *dst, int64_t n) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        dst[k] = src[perm[k]];
}

__device__ __forceinline__ int ordered_key(float f) {
    int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float ordered_val(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff); }

__global__ void k_init_min(int *slot) { *slot = 0x7fffffff; }

__global__ void k_min(const float *S, int64_t n, int *slot) {
    int best = 0x7fffffff;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        best = min(best, ordered_key(S[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) atomicMin(slot, best);
}

// Eq. 3-10, double precision per element.
__global__ void k_normalize(const float *S, float *t, int64_t n, const int *slot, double *mh) {
    double m = (double)ordered_val(*slot);
    double h = log(2.0) / (m * m);
    if (blockIdx.x == 0 && threadIdx.x == 0 && mh) {
        mh[0] = m;
        mh[1] = h;
    }
    __shared__ ff c[kEq310Terms];
    if (threadIdx.x == 0) eq310_coefs(c);
    __syncthreads();
    const float mf = ordered_val(*slot);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        t[i] = eq310_target(S[i], mf, c);
}

__global__ void k_state_init(serbf_state *st, double lr) {
    serbf_state z;
    memset(&z, 0, sizeof(z));
    z.lr = lr;
    z.alpha = 1.0;
    z.beta = 0.0;
    *st = z;
}

int grid_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

}  // namespace

namespace serbf {
int launch_exscan_i64(int64_t *a, int64_t n, int64_t *tiles, cudaStream_t s) {
    static_assert(kScanThreads * kScanPer == kScanTile, "elements per block");
    const int64_t nt = n > 0 ? (n + kScanTile - 1) / kScanTile : 1;
    launch_pdl(k_scan_tile<true>, dim3((unsigned)nt), dim3(kScanThreads), 0, s, a, n, tiles);
    launch_pdl(k_scan_sums, dim3(1), dim3(1024), 0, s, tiles, nt);
    launch_pdl(k_scan_tile<false>, dim3((unsigned)nt), dim3(kScanThreads), 0, s, a, n, tiles);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}
}  // namespace serbf

extern "C" {

const char *serbf_version(void) { return "serbf 0.4.2 (sm_103a)"; }

const char *serbf_status_string(int code) {
    switch (code) {
        case SERBF_OK: return "ok";
        case SERBF_EINVAL: return "invalid argument";
        case SERBF_ENOMEM: return "workspace too small";
        case SERBF_ECAPACITY: return "capacity exceeded";
        case SERBF_ECUDA: return "CUDA error";
        case SERBF_ETIMEOUT: return "device wait timed out";
        default: return "unknown status";
    }
}

int serbf_config_default(serbf_config *c) {
    if (!c) return SERBF_EINVAL;
    memset(c, 0, sizeof(*c));
    c->eps = 1e-7;
    c->tau1 = 0.9;
    c->tau2 = 1.1;
    c->tau_m = 0.02;
    c->tau_d = 0.01;
    c->tau_l1 = 5.0;
    c->tau_l2 = 0.5;
    c->lr = 0.01;
    c->lr_p2 = 1e-3;
    c->lr_min = 1e-5;
    c->beta1 = 0.9;
    c->beta2 = 0.999;
    c->adam_eps = 1e-8;
    c->topk_frac = 0.01;
    c->add_radius = 0.0;
    c->dbar_min = 0.0;
    c->k_l1 = 50;
    c->k_l2 = 10;
    c->T_e = 1600;
    c->M_e = 2000;
    c->kahan = 0;
    c->epoch_steps = 1;
    return SERBF_OK;
}

size_t serbf_workspace_struct_size(void) { return sizeof(serbf_workspace); }

int serbf_workspace_bytes(const serbf_ws_sizes *sz, size_t *bytes) {
    if (!sizes_ok(sz) || !bytes) return SERBF_EINVAL;
    serbf_workspace tmp;
    memset(&tmp, 0, sizeof(tmp));
    Carver c{nullptr};
    carve(c, &tmp, sz);
    *bytes = align_up(c.off, 256);
    return SERBF_OK;
}

int serbf_workspace_init(serbf_workspace *ws, void *dev, size_t bytes, const serbf_ws_sizes *sz) {
    if (!ws || !dev || !sizes_ok(sz)) return SERBF_EINVAL;
    if (((uintptr_t)dev) % 256) return SERBF_EINVAL;
    size_t need;
    serbf_workspace_bytes(sz, &need);
    if (bytes < need) return SERBF_ENOMEM;
    memset(ws, 0, sizeof(*ws));
    ws->magic = kMagic;
    ws->base = (char *)dev;
    ws->bytes = bytes;
    ws->sz = *sz;
    Carver c{(char *)dev};
    carve(c, ws, sz);
    if (cudaMemset(ws->status, 0, 16 * sizeof(int32_t)) != cudaSuccess) return SERBF_ECUDA;
    if (cudaMemset(ws->needed, 0, 4 * sizeof(long long)) != cudaSuccess) return SERBF_ECUDA;
    if (cudaMemset(ws->counters, 0, 16 * sizeof(uint32_t)) != cudaSuccess) return SERBF_ECUDA;
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return SERBF_ECUDA;
        if (cudaDeviceGetAttribute(&ws->sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return SERBF_ECUDA;
    }
    if (cudaMemset(ws->add_info, 0, 16 * sizeof(int32_t)) != cudaSuccess) return SERBF_ECUDA;
    if (cudaMemset(ws->sel_hist, 0, kSelBins * sizeof(uint32_t)) != cudaSuccess) return SERBF_ECUDA;
    if (cudaMemset(ws->cell_max, 0, 4 * sizeof(uint32_t)) != cudaSuccess) return SERBF_ECUDA;
    if (cudaMemset(ws->sel_ctl, 0, 16 * sizeof(uint32_t)) != cudaSuccess) return SERBF_ECUDA;
    if (cudaMemset(ws->adj_fix, 0, sizeof(unsigned long long) * 10 * (size_t)sz->max_kernels) != cudaSuccess)
        return SERBF_ECUDA;
    if (cudaMemset(ws->adj_pairs, 0, sizeof(unsigned long long) * 8) != cudaSuccess) return SERBF_ECUDA;
    if (cudaStreamCreateWithFlags(&ws->aux, cudaStreamNonBlocking) != cudaSuccess) return SERBF_ECUDA;
    if (cudaEventCreateWithFlags(&ws->ev_fork, cudaEventDisableTiming) != cudaSuccess) return SERBF_ECUDA;
    if (cudaEventCreateWithFlags(&ws->ev_join, cudaEventDisableTiming) != cudaSuccess) return SERBF_ECUDA;
    if (cudaDeviceSynchronize() != cudaSuccess) return SERBF_ECUDA;
    return SERBF_OK;
}

int serbf_workspace_release(serbf_workspace *ws) {
    if (!ws || ws->magic != kMagic) return SERBF_EINVAL;
    int rc = SERBF_OK;
    if (ws->aux && cudaStreamSynchronize(ws->aux) != cudaSuccess) rc = SERBF_ECUDA;
    if (ws->aux && cudaStreamDestroy(ws->aux) != cudaSuccess) rc = SERBF_ECUDA;
    if (ws->ev_fork && cudaEventDestroy(ws->ev_fork) != cudaSuccess) rc = SERBF_ECUDA;
    if (ws->ev_join && cudaEventDestroy(ws->ev_join) != cudaSuccess) rc = SERBF_ECUDA;
    ws->aux = nullptr;
    ws->ev_fork = ws->ev_join = nullptr;
    ws->magic = 0;
    return rc;
}

int serbf_status(serbf_workspace *ws, int32_t *flags, int64_t needed[4], int clear, void *stream) {
    if (!ws || ws->magic != kMagic) return SERBF_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    int32_t f = 0;
    long long nd[4] = {0, 0, 0, 0};
    if (cudaMemcpyAsync(&f, ws->status, sizeof(int32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return SERBF_ECUDA;
    if (cudaMemcpyAsync(nd, ws->needed, sizeof(nd), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return SERBF_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return SERBF_ECUDA;
    if (flags) *flags = f;
    if (needed)
        for (int k = 0; k < 4; ++k) needed[k] = nd[k];
    if (clear) {
        if (cudaMemsetAsync(ws->status, 0, sizeof(int32_t), s) != cudaSuccess) return SERBF_ECUDA;
        if (cudaMemsetAsync(ws->needed, 0, 4 * sizeof(long long), s) != cudaSuccess) return SERBF_ECUDA;
    }
    return f ? SERBF_ECAPACITY : SERBF_OK;
}

int serbf_state_init(serbf_state *st_dev, const serbf_config *cfg, void *stream) {
    if (!st_dev || !cfg) return SERBF_EINVAL;
    k_state_init<<<1, 1, 0, (cudaStream_t)stream>>>(st_dev, cfg->lr);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

int serbf_normalize_sdf(const float *S, float *t, int64_t n, double *mh_dev, serbf_workspace *ws,
                        void *stream) {
    SERBF_TRACE();
    if (!S || !t || n <= 0 || !ws || ws->magic != kMagic) return SERBF_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    int *slot = ws->status + 8;
    k_init_min<<<1, 1, 0, s>>>(slot);
    k_min<<<grid_for(n, 256), 256, 0, s>>>(S, n, slot);
    k_normalize<<<grid_for(n, 256), 256, 0, s>>>(S, t, n, slot, mh_dev);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

int serbf_gather(const float *src, const uint32_t *perm, float *dst, int64_t n, void *stream) {
    if (n < 0 || (n > 0 && (!src || !perm || !dst))) return SERBF_EINVAL;
    if (n == 0) return SERBF_OK;
    k_gather<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(src, perm, dst, n);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

}  // extern "C"
