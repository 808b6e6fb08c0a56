// Point-major forward (Eq. 3-26) over the support pairs of Eq. 3-15-1, the
// point filter of Eq. 3-18 and the loss terms of Eq. 3-19.
//
// Work item = up to two (several warps per item) or four (one warp per item)
// consecutive 32-point tiles of one super cell; each lane holds one point of
// each tile.  The warp streams
// its super cell's candidate list (ascending kernel index), keeps the kernels
// whose support reaches the item's bounding box (one candidate per lane,
// ballot), and stages their records in a per-warp shared-memory ring, in
// pairs.  Each batch of 32 staged kernels is then evaluated with broadcast
// 16-byte loads and packed f32x2 arithmetic (two kernels per instruction,
// two or four points per lane), so every shared-memory load serves four or
// eight pairs.  A kernel whose support covers the whole box skips the
// predicate; otherwise every lane applies the exact support predicate to its
// own points, so the pairs summed are exactly the point-major neighbour rows.
//
// What bounds it is the instructions issued: pair arithmetic is 40 % of them,
// the rest scans, stages, filters and flushes per item.  Four tiles per item
// halve that rest per point and widen the item box (a few more pairs outside
// the support); with one warp per item that gains (9.4 M points 2118 -> 2070 us,
// 16 fields 844 -> 704 us for the fused call), with several it does not (64^3 +
// 32^3 points 60 -> 64 us with four, 128^3 292 -> 318 with two), so they keep two.
// The tiles follow from the warps alone, so a field in a batch gets the bits it
// gets by itself.
//
// Persistent blocks take items heaviest first (order from the costs measured
// by the previous launch) to keep the tail short; the warps of a block split
// an item's candidate list and combine their sums in a fixed order.
#include <math.h>
#include <string.h>

#include "common.cuh"
#include "form_bound.cuh"
#include "warps_rule.cuh"

using namespace serbf;

namespace {

struct FwdArgs {
    const float *x, *y, *z, *t;
    const float4 *tile_lo, *tile_hi;
    const uint32_t *slist, *scnt;
    const float4 *kfwd;
    const uint4 *order_rec;  // item records, heaviest class first (stable)
    uint8_t *item_class;     // cost class of each item, for the next order
    uint32_t *sched;         // mean cost of the last launch
    unsigned long long *sched_total;
    unsigned long long *adj_fix;    // fixed-point moments (fused adjoint)
    unsigned long long *adj_pairs;  // adjoint pair count (fused adjoint)
    int64_t nitems;
    int scap;
    float tau1, tau2;  // tau1 rounded down, tau2 rounded up to float: exact double decisions
    float *psi, *err;
    uint8_t *mask;
    FwdPart *part;        // one partial per tile
    uint32_t *item_next;  // next work item to take (zero between launches)
    uint32_t *exit_count; // blocks that have exited (zero between launches)
    int32_t *status;      // device status flags
};

constexpr int kTouch = 256;  // kernels an item's warps remember for its adjoint (more: re-scan the list)
constexpr int kNz = kMostTiles * kTile;

// Two float32 lanes in one 64-bit register: the packed f32x2 arithmetic of
// sm_100+ does two IEEE round-to-nearest operations per instruction, each
// bit-identical to its scalar counterpart.
typedef unsigned long long f2;

__device__ __forceinline__ f2 f2_pack(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(f2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Staged kernels are stored in pairs, interleaved so that one 16-byte load
// gives the same field of both kernels (a packed f32x2 operand).  Field v of
// the kernel in ring slot s is at float 24 (s / 2) + 2 v + s % 2, with fields
// cx, cy, cz, r2, Q11, Q22, Q33, a = w|w|, 2Q12, 2Q13, 2Q23 (v = 0 .. 10).
constexpr int kPairFloats = 24;

__device__ __forceinline__ void stage(float *ring, int slot, float4 k0, float4 k1, float4 k2) {
    float *b = ring + kPairFloats * (slot >> 1) + (slot & 1);
    b[0] = k0.x;
    b[2] = k0.y;
    b[4] = k0.z;
    b[6] = k0.w;
    b[8] = k1.x;
    b[10] = k1.y;
    b[12] = k1.z;
    b[14] = k1.w;
    b[16] = k2.x;
    b[18] = k2.y;
    b[20] = k2.z;
}

// The empty partner of an odd last kernel: q = 0, a = 0 and r2 < 0, so it
// adds exactly zero and is never counted.
__device__ __forceinline__ void stage_empty(float *ring, int slot) {
    float *b = ring + kPairFloats * (slot >> 1) + (slot & 1);
#pragma unroll
    for (int v = 0; v < 11; ++v) b[2 * v] = 0.f;
    b[6] = -1.f;
}

// Squared distance from c to the farthest corner of a box, rounded so that
// it is never below the support_d2 of any point inside the box:
// box_far_d2 < r2 means every point of the box is in the support.
__device__ __forceinline__ float box_far_d2(float cx, float cy, float cz, float4 lo, float4 hi) {
    const float ax = fmaxf(__fsub_rn(cx, lo.x), __fsub_rn(hi.x, cx));
    const float ay = fmaxf(__fsub_rn(cy, lo.y), __fsub_rn(hi.y, cy));
    const float az = fmaxf(__fsub_rn(cz, lo.z), __fsub_rn(hi.z, cz));
    return support_d2(ax, ay, az);
}

// box_d2 and box_far_d2 from the same differences: with a = lo - c and b =
// c - hi on an axis, the near distance is max(a, b, 0) and the far one
// max(-a, -b), the values of the two functions bit for bit (rounding is
// symmetric; a NaN centre gives near 0).
__device__ __forceinline__ void box_near_far_d2(float cx, float cy, float cz, float4 lo, float4 hi, float &near2,
                                                float &far2) {
    const float ax = __fsub_rn(lo.x, cx), ay = __fsub_rn(lo.y, cy), az = __fsub_rn(lo.z, cz);
    const float bx = __fsub_rn(cx, hi.x), by = __fsub_rn(cy, hi.y), bz = __fsub_rn(cz, hi.z);
    near2 = support_d2(fmaxf(fmaxf(ax, bx), 0.f), fmaxf(fmaxf(ay, by), 0.f), fmaxf(fmaxf(az, bz), 0.f));
    far2 = support_d2(fminf(ax, bx), fminf(ay, by), fminf(az, bz));
}

// npairs staged kernel pairs from pair index pb against the lane's points.
// NP: those that take part, of NT (an item of a sparse super cell may have
// fewer tiles).  PARTIAL: the support only partly covers the item box, so each
// pair takes the exact Eq. 3-15-1 predicate (the operations of support_d2,
// packed: fma(dz, dz, fma(dy, dy, fl(dx dx))) < r2).
template <bool PARTIAL, int UNROLL, int NP, int NT>
__device__ __forceinline__ void eval_pairs(const float *ring, int pb, int npairs, const f2 (&P)[NT][3], f2 (&acc)[NT],
                                           uint32_t (&n)[NT]) {
#pragma unroll UNROLL
    for (int q = 0; q < npairs; ++q) {
        const ulonglong2 *r = reinterpret_cast<const ulonglong2 *>(ring + kPairFloats * (pb + q));
        const ulonglong2 F0 = r[0], F1 = r[1], F2 = r[2], F3 = r[3], F4 = r[4], F5 = r[5];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const f2 dx = f2_sub(P[p][0], F0.x), dy = f2_sub(P[p][1], F0.y), dz = f2_sub(P[p][2], F1.x);
            const f2 zz = f2_mul(dz, dz);
            // q = dv^T Q dv (log2 units): dx (Q11 dx + 2Q12 dy + 2Q13 dz) + dy (Q22 dy + 2Q23 dz) + Q33 dz^2
            const f2 ra = f2_fma(F4.y, dz, f2_fma(F4.x, dy, f2_mul(F2.x, dx)));
            const f2 rb = f2_fma(F5.x, dz, f2_mul(F2.y, dy));
            const f2 qv = f2_fma(F3.x, zz, f2_fma(dy, rb, f2_mul(dx, ra)));
            float q0, q1;
            f2_unpack(qv, q0, q1);
            float e0 = ex2_approx(-q0), e1 = ex2_approx(-q1);
            if (PARTIAL) {
                const f2 d2 = f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
                float d0, d1, r0, r1;
                f2_unpack(d2, d0, d1);
                f2_unpack(F1.y, r0, r1);
                const bool i0 = d0 < r0, i1 = d1 < r1;
                e0 = i0 ? e0 : 0.f;
                e1 = i1 ? e1 : 0.f;
                n[p] += (uint32_t)i0 + (uint32_t)i1;
            }
            acc[p] = f2_fma(F3.y, f2_pack(e0, e1), acc[p]);
        }
    }
}

template <bool PARTIAL, int UNROLL, int NT>
__device__ __forceinline__ void eval_staged(int ntl, const float *ring, int pb, int npairs, const f2 (&P)[NT][3],
                                            f2 (&acc)[NT], uint32_t (&n)[NT]) {
    if constexpr (NT > 2) {
        if (ntl > 2)
            eval_pairs<PARTIAL, 1, NT>(ring, pb, npairs, P, acc, n);  // four points are enough independent chains
        else
            eval_pairs<PARTIAL, 1, 2>(ring, pb, npairs, P, acc, n);
    } else {
        eval_pairs<PARTIAL, UNROLL, 2>(ring, pb, npairs, P, acc, n);
    }
}

// Whole-warp reductions in one instruction (redux.sync, sm_100 family): exact
// for integers; min / max of floats select one of the inputs, so the result
// does not depend on the order.
__device__ __forceinline__ uint32_t redux_add(uint32_t v) {
    uint32_t r;
    asm volatile("redux.sync.add.u32 %0, %1, 0xffffffff;" : "=r"(r) : "r"(v));
    return r;
}
__device__ __forceinline__ uint32_t redux_max_u32(uint32_t v) {
    uint32_t r;
    asm volatile("redux.sync.max.u32 %0, %1, 0xffffffff;" : "=r"(r) : "r"(v));
    return r;
}
// Partial of a group of tiles: the loss sum in double (the global loss
// reduction runs in FP64; a tile's own sum of 32 squares is float-float).
struct FwdGPart {
    double l2;
    float maxe;
    uint32_t cnt;
    unsigned long long pairs;
};
static_assert(sizeof(FwdGPart) == sizeof(FwdPart), "group partials reuse the tile-partial storage");

__device__ __forceinline__ double part_l2(const FwdPart *p, uint32_t q) {
    return (double)__ldcg(&p[q].l2hi) + (double)__ldcg(&p[q].l2lo);
}
__device__ __forceinline__ double part_l2(const FwdGPart *p, uint32_t q) { return __ldcg(&p[q].l2); }

// Fixed-order warp reduction of partials [b, e) (of tiles or of groups) into one.
template <typename P>
__device__ __forceinline__ FwdGPart reduce_parts(const P *p, uint32_t b, uint32_t e, int lane) {
    double l = 0.0;
    float mx = 0.f;
    unsigned long long c = 0, pr = 0;
#pragma unroll 4
    for (uint32_t q = b + lane; q < e; q += 32) {
        l += part_l2(p, q);
        mx = fmaxf(mx, __ldcg(&p[q].maxe));
        c += __ldcg(&p[q].cnt);
        pr += __ldcg(&p[q].pairs);
    }
    l = warp_sum(l);
    mx = warp_max(mx);
    c = warp_sum(c);
    pr = warp_sum(pr);
    return FwdGPart{l, mx, (uint32_t)c, pr};
}

// Loss terms of one tile, stored as the tile's partial (lane order within the
// tile).  The partials are reduced in tile order after the launch, so the
// totals do not depend on which warp handled which tile. 
__device__ __forceinline__ void finish_tile(const FwdArgs &a, uint32_t t, float l2, float mx_l, uint32_t cnt_l,
                                            uint32_t pairs_l, int lane) {
    const ff l2s = warp_sum_ff(ff{l2, 0.f});
    const float mx = redux_max(mx_l);
    const uint32_t cnt = redux_add(cnt_l), pr = redux_add(pairs_l);
    if (lane == 0) a.part[t] = FwdPart{l2s.hi, l2s.lo, mx, cnt, (unsigned long long)pr};
}

// Loss terms of an item's ntl tiles in one reduction (a lane's squares are
// summed in float-float first), stored as the first tile's partial; the other
// tiles' are zero.
__device__ __forceinline__ void finish_item(const FwdArgs &a, uint32_t t, int ntl, ff l2, float mx_l, uint32_t cnt_l,
                                            uint32_t pairs_l, int lane) {
    const ff l2s = warp_sum_ff(l2);
    const float mx = redux_max(mx_l);
    const uint32_t cnt = redux_add(cnt_l), pr = redux_add(pairs_l);
    if (lane == 0) a.part[t] = FwdPart{l2s.hi, l2s.lo, mx, cnt, (unsigned long long)pr};
    if (lane > 0 && lane < ntl) a.part[t + lane] = FwdPart{0.f, 0.f, 0.f, 0u, 0ull};
}

// Eq. 3-18 filter of one point: whether it is in id_all, and its residual.
__device__ __forceinline__ bool point_residual(const FwdArgs &a, bool valid, float t, float ps, float &e) {
    const bool m0 = (a.tau1 < t) && (t < a.tau2);
    const bool m1 = (t <= a.tau1) && (ps > a.tau1);
    const bool m2 = (t >= a.tau2) && (ps < a.tau2);
    const bool mk = valid && (m0 || m1 || m2);
    e = mk ? __fsub_rn(ps, t) : 0.f;
    return mk;
}

// The outputs of one point; returns its residual and loss contributions.
__device__ __forceinline__ float point_out(const FwdArgs &a, int64_t i, bool valid, float t, float ps, uint32_t np,
                                           float &l2, float &mx, uint32_t &cnt, uint32_t &pairs) {
    l2 = 0.f;
    mx = 0.f;
    cnt = 0u;
    pairs = 0u;
    if (!valid) return 0.f;
    float e;
    const bool mk = point_residual(a, valid, t, ps, e);
    a.psi[i] = ps;
    a.err[i] = e;
    a.mask[i] = (uint8_t)mk;
    pairs = np;
    if (mk) {
        l2 = e * e;
        mx = fabsf(e);
        cnt = 1u;
    }
    return e;
}

// Item geometry shared by the warps of a block: tiles t0 .. t0 + ntl - 1 of
// super cell sup, np points from i0 (a lane's points: i0 + lane + 32 k).
struct ItemInfo {
    uint32_t t0, sup;
    int ntl, np;
    int64_t i0;
};

// Decode an item record (first tile, super cell, first point, points - 1 | item << 7).
__device__ __forceinline__ ItemInfo item_info(uint4 r) {
    ItemInfo it;
    it.np = (int)(r.w & 127u) + 1;
    it.t0 = r.x;
    it.sup = r.y;
    it.ntl = (it.np + kTile - 1) / kTile;
    it.i0 = (int64_t)r.z;
    return it;
}

__device__ __forceinline__ float4 box_min(float4 a, float4 b) {
    return make_float4(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z), 0.f);
}
__device__ __forceinline__ float4 box_max(float4 a, float4 b) {
    return make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z), 0.f);
}

// Warp w's share [b0, b1) of a list of n candidates: an equal run.  (Chunks
// of 32 dealt round-robin gave a warp up to twice another's candidates when a
// list holds one or two chunks per warp, and the others waited at the barrier.)
template <int G>
__device__ __forceinline__ void share_of(int n, int w, int &b0, int &b1) {
    const int per = (n + G - 1) / G;
    b0 = G > 1 ? w * per : 0;
    b1 = G > 1 ? min(n, b0 + per) : n;
}

// One warp's share of a work item: its run of the super cell's list is
// filtered against the item box, 32 candidates at a time,
// staged in pairs and evaluated against the lane's points.
// Returns the lane's partial sums and pair counts; *cost gets the warp's
// measured work.
template <int G, int ADJ, int NT>
__device__ __forceinline__ void forward_share(const FwdArgs &a, const ItemInfo &it, int w, float *ringP, float *ringF,
                                              int lane, f2 (&acc)[NT], uint32_t (&n)[NT], uint32_t &cost,
                                              uint32_t *touch, int tcap, int &ntouch) {
    const unsigned lt = (1u << lane) - 1u;
    // invalid lanes carry NaN so the support test fails for them
    const float qnan = __int_as_float(0x7fc00000);
    f2 P[NT][3];
#pragma unroll
    for (int p = 0; p < NT; ++p) {
        const bool v = lane + p * kTile < it.np;
        const int64_t i = it.i0 + lane + p * kTile;
        const float x = v ? a.x[i] : qnan, y = v ? a.y[i] : 0.f, z = v ? a.z[i] : 0.f;
        P[p][0] = f2_pack(x, x);
        P[p][1] = f2_pack(y, y);
        P[p][2] = f2_pack(z, z);
        acc[p] = 0ull;
        n[p] = 0u;
    }
    float4 lo = a.tile_lo[it.t0], hi = a.tile_hi[it.t0];
#pragma unroll
    for (int p = 1; p < NT; ++p)
        if (p < it.ntl) {
            lo = box_min(lo, a.tile_lo[it.t0 + p]);
            hi = box_max(hi, a.tile_hi[it.t0 + p]);
        }
    const uint32_t *lst = a.slist + (size_t)it.sup * a.scap;
    int b0, L;
    share_of<G>(min((int)a.scnt[it.sup], a.scap), w, b0, L);
    int hp = 0, qp = 0, hf = 0, qf = 0;
    uint32_t nfull = 0, npart = 0;
    // software pipeline: records of the next chunk and indices of the one
    // after it are in flight while a chunk is filtered
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t jc = b0 + lane < L ? lst[b0 + lane] : 0u;
    float4 c0 = zero4, c1 = zero4, c2 = zero4;
    if (b0 + lane < L) {
        c0 = a.kfwd[3 * jc];
        c1 = a.kfwd[3 * jc + 1];
        c2 = a.kfwd[3 * jc + 2];
    }
    uint32_t jn = b0 + 32 + lane < L ? lst[b0 + 32 + lane] : 0u;
    int nchunks = 0;
    ntouch = 0;
    for (int b = b0; b < L; b += 32) {
        const float4 k0 = c0, k1 = c1, k2 = c2;
        const uint32_t j = jc;
        const bool live = b + lane < L;
        if (b + 32 + lane < L) {
            c0 = a.kfwd[3 * jn];
            c1 = a.kfwd[3 * jn + 1];
            c2 = a.kfwd[3 * jn + 2];
        }
        jc = jn;
        if (b + 64 + lane < L) jn = lst[b + 64 + lane];
        ++nchunks;
        float near2, far2;
        box_near_far_d2(k0.x, k0.y, k0.z, lo, hi, near2, far2);
        const bool hit = live && near2 < k0.w, full = hit && far2 < k0.w;
        const unsigned ba = __ballot_sync(0xffffffffu, hit), bf = __ballot_sync(0xffffffffu, full), bp = ba & ~bf;
        if (hit) {
            // one store block for both rings: the lane's ring is an offset.  The
            // kernel is bound by the instructions it issues; with a block per
            // ring, a branch around the far test and branches around the
            // adjoint's atomics, the 9.4 M point epoch took 2461 us, without
            // them 2259 us (16 fields: 878 and 775 us).
            const int slot = (full ? hf + qf : hp + qp) + __popc((full ? bf : bp) & lt);
            stage(full ? ringF : ringP, slot & (kQueue - 1), k0, k1, k2);
            if (ADJ) {
                // the kernels that reach the item box, for the adjoint pass
                const int pos = ntouch + __popc(ba & lt);
                if (pos < tcap) touch[pos] = j;
            }
        }
        if (ADJ) ntouch += __popc(ba);
        const int np = __popc(bp), nf = __popc(bf);
        qp += np;
        qf += nf;
        npart += np;
        nfull += nf;
        __syncwarp();
        if (qp >= 32) {
            eval_staged<true, 2>(it.ntl, ringP, hp >> 1, 16, P, acc, n);
            hp ^= 32;
            qp -= 32;
        }
        if (qf >= 32) {
            eval_staged<false, 2>(it.ntl, ringF, hf >> 1, 16, P, acc, n);
            hf ^= 32;
            qf -= 32;
        }
        __syncwarp();
    }
    // leftovers: the head is 0 or 32 and fewer than 32 remain, so they do not
    // wrap; an odd count gets an empty partner
    if (qp & 1) {
        if (lane == 0) stage_empty(ringP, hp + qp);
        __syncwarp();
    }
    if (qf & 1) {
        if (lane == 0) stage_empty(ringF, hf + qf);
        __syncwarp();
    }
    if (qp > 0) eval_staged<true, 1>(it.ntl, ringP, hp >> 1, (qp + 1) >> 1, P, acc, n);
    if (qf > 0) eval_staged<false, 1>(it.ntl, ringF, hf >> 1, (qf + 1) >> 1, P, acc, n);
    __syncwarp();
#pragma unroll
    for (int p = 0; p < NT; ++p) n[p] += nfull;
    // about one unit per filtered candidate, ~6 per fully and ~9 per partly
    // covering kernel and two points of a lane
    cost = 32u * (uint32_t)nchunks + (6u * nfull + 9u * npart) * (NT / 2);
}

// ---------------------------------------------------------------- fused adjoint
// After an item's residuals are known, its points with E != 0 (at most 128 with
// one warp per item, 64 with several; in shared memory in point order, padded to
// an even count) are taken against the kernels that reached the
// item box in the forward filter, kept if their support reaches the box of
// those points: lanes are kernels, each lane loops over the points two at a
// time (packed f32x2) and accumulates the ten moments of its kernel in the
// world frame, Delta = v - c:
//     S0 = sum s,  W1 = sum s Delta,  W2 = sum s Delta Delta^T,  s = phi E,
// with phi = 2^(-Delta^T Q Delta) from the forward's own records (so the
// adjoint evaluates the same quadratic form as the forward).  The kernel
// frame moments of App. A are M1 = R W1 and M2 = R W2 R^T, formed once per
// kernel after the launch.  The item's float partial
// moments go to per-kernel 64-bit fixed-point accumulators (unit 2^-36) by
// integer atomics: integer addition is associative, so the totals do not
// depend on the order in which items finish.

// The nz points in pairs: pair k holds points 2k and 2k + 1 as two 16-byte
// words (x0, x1, y0, y1) and (z0, z1, e0, e1), so one pair of points is two
// 16-byte loads that give the packed operands directly.
struct NzPoints {
    float4 v[kNz];  // kNz / 2 pairs, two words each
    __device__ __forceinline__ float &at(int field, int i) {
        // field 0..3 = x, y, z, e of point i
        float4 &w = v[2 * (i >> 1) + (field >> 1)];
        const int k = 2 * (field & 1) + (i & 1);
        return k == 0 ? w.x : (k == 1 ? w.y : (k == 2 ? w.z : w.w));
    }
};

__device__ __forceinline__ f2 f2_dup(float v) { return f2_pack(v, v); }

// v * 2^36 rounded to the nearest integer (ties to even): the scaling by a
// power of two is exact in float, and one hardware conversion rounds (it was
// 9 % faster on the 256^3 field than an integer-only rounding).  |v| >= 2^26
// does not fit the accumulators' range; the caller flags such a partial
// before converting it.
__device__ __forceinline__ long long to_fix36(float v) {
    return __float2ll_rn(__fmul_rn(v, 68719476736.f));
}

// Predicated 64-bit integer addition without a result (no divergent branch
// around each of the ten moments).
__device__ __forceinline__ void red_add_u64(unsigned long long *p, bool go, long long v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p red.relaxed.gpu.global.add.u64 [%0], %1;\n\t}" ::"l"(p),
                 "l"(v), "r"((int)go)
                 : "memory");
}

// Compensated (Kahan) accumulation of packed pairs: s + v with the lost
// low-order part carried in c.
__device__ __forceinline__ void f2_kadd(f2 &s, f2 &c, f2 v) {
    const f2 y = f2_sub(v, c);
    const f2 t = f2_add(s, y);
    c = f2_sub(f2_sub(t, s), y);
    s = t;
}

// A batch of cnt <= 32 kernels from queue slot head: all nz points of the
// item (nc) against each kernel.  A short batch spreads each kernel over
// L = 2, 4 or 8 neighbouring lanes (cnt <= 16, 8, 4) that take every L-th
// point pair; their moments are combined with xor shuffles within the group
// (a fixed order for a given cnt) before the atomics, so short batches do
// not leave most lanes idle.  KAHAN: compensated per-lane sums.
template <bool KAHAN>
__device__ __forceinline__ void adjoint_batch(const FwdArgs &a, const uint32_t *q, int head, int cnt,
                                              const NzPoints &nz, int nc, int lane) {
    const int sh = cnt > 16 ? 0 : (cnt > 8 ? 1 : (cnt > 4 ? 2 : 3));
    const int L = 1 << sh, kl = lane >> sh, sub = lane & (L - 1);
    const bool act = kl < cnt;  // whole groups of L lanes are inactive together
    const uint32_t j = q[(head + (act ? kl : 0)) & (kQueue - 1)];
    const float4 k0 = a.kfwd[3 * j], k1 = a.kfwd[3 * j + 1], k2 = a.kfwd[3 * j + 2];
    const f2 cx = f2_dup(k0.x), cy = f2_dup(k0.y), cz = f2_dup(k0.z);
    const f2 q11 = f2_dup(k1.x), q22 = f2_dup(k1.y), q33 = f2_dup(k1.z);
    const f2 q12 = f2_dup(k2.x), q13 = f2_dup(k2.y), q23 = f2_dup(k2.z);  // 2 Q12, 2 Q13, 2 Q23
    f2 acc[10], cmp[KAHAN ? 10 : 1];
#pragma unroll
    for (int r = 0; r < 10; ++r) acc[r] = 0ull;
#pragma unroll
    for (int r = 0; r < (KAHAN ? 10 : 1); ++r) cmp[r] = 0ull;
    // nc <= 128: with its range in sight the loop counts in fewer instructions
    // (9.4 M points 2066 -> 2046 us an epoch)
    static_assert(kNz < 256, "residual points of an item");
    const int cntp = act ? (int)(((uint32_t)nc & 255u) + 1u) >> 1 : 0;
#pragma unroll 4
    for (int pp = sub; pp < cntp; pp += L) {
        const int i = 2 * pp;
        const ulonglong2 wa = *reinterpret_cast<const ulonglong2 *>(&nz.v[i]);
        const ulonglong2 wb = *reinterpret_cast<const ulonglong2 *>(&nz.v[i + 1]);
        const f2 px = wa.x, py = wa.y, pz = wb.x, pe = wb.y;
        const f2 dx = f2_sub(px, cx), dy = f2_sub(py, cy), dz = f2_sub(pz, cz);
        const f2 zz = f2_mul(dz, dz);
        // q = Delta^T Q Delta (log2 units), the forward's operation order
        const f2 ra = f2_fma(q13, dz, f2_fma(q12, dy, f2_mul(q11, dx)));
        const f2 rb = f2_fma(q23, dz, f2_mul(q22, dy));
        const f2 qv = f2_fma(q33, zz, f2_fma(dy, rb, f2_mul(dx, ra)));
        float q0, q1;
        f2_unpack(qv, q0, q1);
        float e0 = ex2_approx(-q0), e1 = ex2_approx(-q1);
        // Eq. 3-15-1, the operations of support_d2, packed
        const f2 d2 = f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
        float d0, d1;
        f2_unpack(d2, d0, d1);
        const bool i0 = d0 < k0.w, i1 = d1 < k0.w;
        e0 = i0 ? e0 : 0.f;
        e1 = i1 ? e1 : 0.f;
        const f2 sv = f2_mul(f2_pack(e0, e1), pe);
        const f2 sx = f2_mul(sv, dx), sy = f2_mul(sv, dy), sz = f2_mul(sv, dz);
        if (KAHAN) {
            f2_kadd(acc[0], cmp[0], sv);
            f2_kadd(acc[1], cmp[1], sx);
            f2_kadd(acc[2], cmp[2], sy);
            f2_kadd(acc[3], cmp[3], sz);
            f2_kadd(acc[4], cmp[4], f2_mul(sx, dx));
            f2_kadd(acc[5], cmp[5], f2_mul(sx, dy));
            f2_kadd(acc[6], cmp[6], f2_mul(sx, dz));
            f2_kadd(acc[7], cmp[7], f2_mul(sy, dy));
            f2_kadd(acc[8], cmp[8], f2_mul(sy, dz));
            f2_kadd(acc[9], cmp[9], f2_mul(sz, dz));
        } else {
            acc[0] = f2_add(acc[0], sv);
            acc[1] = f2_add(acc[1], sx);
            acc[2] = f2_add(acc[2], sy);
            acc[3] = f2_add(acc[3], sz);
            acc[4] = f2_fma(sx, dx, acc[4]);
            acc[5] = f2_fma(sx, dy, acc[5]);
            acc[6] = f2_fma(sx, dz, acc[6]);
            acc[7] = f2_fma(sy, dy, acc[7]);
            acc[8] = f2_fma(sy, dz, acc[8]);
            acc[9] = f2_fma(sz, dz, acc[9]);
        }
    }
    float v[10];
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        float lo, hi;
        f2_unpack(acc[r], lo, hi);
        if (KAHAN) {
            // the two halves and their compensations, as a float-float sum
            float clo, chi;
            f2_unpack(cmp[r], clo, chi);
            const ff t = ff_add(two_sum(lo, -clo), two_sum(hi, -chi));
            v[r] = t.hi + t.lo;
        } else {
            v[r] = lo + hi;
        }
    }
    for (int o = 1; o < L; o <<= 1) {
#pragma unroll
        for (int r = 0; r < 10; ++r) v[r] += __shfl_xor_sync(0xffffffffu, v[r], o);
    }
    if (act && sub == 0) {
        // a partial at or beyond 2^26 (or not finite) does not fit the
        // fixed-point range: flag it (never taken in a healthy fit)
        bool out = false;
#pragma unroll
        for (int r = 0; r < 10; ++r) out |= !(fabsf(v[r]) < 67108864.f);
        if (out) atomicOr(a.status, SERBF_FLAG_FIX_RANGE);
        unsigned long long *o = a.adj_fix + 10 * (size_t)j;
#pragma unroll
        for (int r = 0; r < 10; ++r)
            red_add_u64(o + r, v[r] != 0.f, to_fix36(v[r]));
    }
}

// One warp's share of an item's adjoint: the kernels this warp found
// reaching the item box (or, if it found more than tcap, its candidate
// chunks of the super cell's list again), filtered against the nz box.  A
// kernel whose form is so large over that box that every moment would be
// converted to a fixed-point zero is left out as well: it would add nothing
// (supports are balls of the longest axis, so about a quarter of the support
// pairs of kernels with axes of 1 : 4 lie there; the kernels that stay may form
// a shorter last batch, which other lanes share, and round otherwise).  The
// test stands here and not in the forward's scan, where every candidate would
// pay for it: an epoch of 9.4 M points and 16384 kernels took 2560 us without
// it, 2462 us with it here, 2533 us with it there.
template <int G, bool KAHAN>
__device__ __forceinline__ void adjoint_share(const FwdArgs &a, const ItemInfo &it, int w, const NzPoints &nz,
                                              int nc, float4 lo, float4 hi, const uint32_t *touch, int ntouch, int tcap,
                                              float emax, uint32_t *q, int lane, uint32_t &cost) {
    const unsigned lt = (1u << lane) - 1u;
    const uint32_t *lst = a.slist + (size_t)it.sup * a.scap;
    const bool listed = ntouch <= tcap;
    int b0 = 0, L = ntouch;
    if (!listed) share_of<G>(min((int)a.scnt[it.sup], a.scap), w, b0, L);
    const float4 mid = make_float4(0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y), 0.5f * (lo.z + hi.z), 0.f);
    const float ex = hi.x - lo.x, ey = hi.y - lo.y, ez = hi.z - lo.z;
    const float hd = 0.5001f * sqrtf(fmaf(ex, ex, fmaf(ey, ey, ez * ez)));
    const float qlim = form_limit(emax, nc);
    int head = 0, qn = 0, nk = 0;
    for (int b = b0; b < L; b += 32) {
        const bool live = b + lane < L;
        const uint32_t j = live ? (listed ? touch[b + lane] : lst[b + lane]) : 0u;
        bool hit = false;
        if (live) {
            const float4 k0 = a.kfwd[3 * j], k1 = a.kfwd[3 * j + 1], k2 = a.kfwd[3 * j + 2];
            hit = box_d2(k0.x, k0.y, k0.z, lo, hi) < k0.w && !(form_floor(k0, k1, k2, mid, hd) > qlim);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, hit);
        if (hit) q[(head + qn + __popc(bal & lt)) & (kQueue - 1)] = j;
        qn += __popc(bal);
        nk += __popc(bal);
        __syncwarp();
        if (qn >= 32) {
            adjoint_batch<KAHAN>(a, q, head, 32, nz, nc, lane);
            head = (head + 32) & (kQueue - 1);
            qn -= 32;
            __syncwarp();
        }
    }
    if (qn > 0) adjoint_batch<KAHAN>(a, q, head, qn, nz, nc, lane);
    __syncwarp();
    cost += (uint32_t)(nk * nc) / 4u + 32u;
}

// The nz points of one 32-point tile (lanes = points), compacted in lane
// order from slot `base`; returns their count.
__device__ __forceinline__ int nz_tile(NzPoints &nzp, int base, bool nz, float x, float y, float z, float e, int lane) {
    const unsigned bal = __ballot_sync(0xffffffffu, nz);
    if (nz) {
        const int i = base + __popc(bal & ((1u << lane) - 1u));
        nzp.at(0, i) = x;
        nzp.at(1, i) = y;
        nzp.at(2, i) = z;
        nzp.at(3, i) = e;
    }
    return __popc(bal);
}

// Pads a run of nz points that ends at slot `end` to an even count: a copy of
// the last point with E = 0 (finite, adds zero, not counted).  One lane, after
// a __syncwarp.
__device__ __forceinline__ void nz_pad(NzPoints &nzp, int end) {
    nzp.at(0, end) = nzp.at(0, end - 1);
    nzp.at(1, end) = nzp.at(1, end - 1);
    nzp.at(2, end) = nzp.at(2, end - 1);
    nzp.at(3, end) = 0.f;
}

// A lane's share of the box of the nz points (empty: +inf / -inf), and the
// warp's box of the lanes' shares.
__device__ __forceinline__ void nz_grow(float4 &lo, float4 &hi, bool nz, float x, float y, float z) {
    if (nz) {
        lo = make_float4(fminf(lo.x, x), fminf(lo.y, y), fminf(lo.z, z), 0.f);
        hi = make_float4(fmaxf(hi.x, x), fmaxf(hi.y, y), fmaxf(hi.z, z), 0.f);
    }
}
__device__ __forceinline__ void nz_box(float4 &lo, float4 &hi) {
    lo = make_float4(redux_min(lo.x), redux_min(lo.y), redux_min(lo.z), 0.f);
    hi = make_float4(redux_max(hi.x), redux_max(hi.y), redux_max(hi.z), 0.f);
}

// ---------------------------------------------------------------- scheduling
// Heavy-first order: blocks claim positions of order_rec, which lists the
// items by the cost class the previous launch measured, heaviest first and
// in natural (spatially coherent) order within a class.  Every launch files
// each item's class for the next order.  Each item is evaluated exactly once
// whatever the order, and the loss partials are reduced by tile index, so
// the order never changes a result.
__device__ __forceinline__ uint4 resolve(const FwdArgs &a, uint32_t k) {
    return (int64_t)k < a.nitems ? a.order_rec[k] : make_uint4(~0u, 0u, 0u, 0u);  // x = ~0: none left
}

// Class of a measured cost: 0 below mean / 4, then about one class per half
// octave up to 7 at 4 x mean and above (all in class 3 before a mean exists).
__device__ __forceinline__ int cost_class(uint32_t c, uint32_t mean) {
    if (mean == 0) return 3;
    const uint64_t c4 = 4ull * c;
    int k = 0;
    k += c4 >= mean;         // >= mean / 4
    k += c4 >= 2ull * mean;  // >= mean / 2
    k += c4 >= 3ull * mean;  // >= 0.75 mean
    k += c4 >= 4ull * mean;  // >= mean
    k += c4 >= 6ull * mean;  // >= 1.5 mean
    k += c4 >= 8ull * mean;  // >= 2 mean
    k += c4 >= 16ull * mean; // >= 4 mean
    return k;
}

// Files an item's class by its measured cost.
__device__ __forceinline__ void note_cost(const FwdArgs &a, uint32_t mean, uint4 rec, uint32_t c) {
    const uint32_t item = rec.w >> 7;
    const int cls = cost_class(c, mean);
    a.item_class[item] = (uint8_t)cls;
    atomicAdd(a.sched_total, (unsigned long long)c);
}

// Last block out: records the mean cost and resets the claim counters.
__device__ __forceinline__ void sched_finish(const FwdArgs &a) {
    __threadfence();
    if (atomicAdd(a.exit_count, 1u) != gridDim.x - 1) return;
    __threadfence();
    const unsigned long long tot = __ldcg(a.sched_total);
    const unsigned long long mean = a.nitems > 0 ? tot / (unsigned long long)a.nitems : 0ull;
    a.sched[0] = (uint32_t)min(mean, 0xffffffffull);
    *a.sched_total = 0ull;
    *a.item_next = 0u;
    *a.exit_count = 0u;
}

// A batch of fields advanced by one launch: the fields' arguments in device
// memory and one order over all their work items, heaviest class first and by
// field within a class (classes are relative to the mean cost of all items, so
// they compare across fields).  Blocks claim positions of that order from one
// counter.  Entry e = (7 - class) nfields + field of the table: its first
// position in the order, and its first place in the field's own order.  (Taken
// field after field, the last field's heavy items came last and the SMs were
// busy 73 % of the launch for 16 fields.)
struct FwdBatch {
    const FwdArgs *args;
    const uint32_t *pos;    // kCostClasses x nfields + 1
    const uint32_t *place;  // kCostClasses x nfields
    int nfields;
    uint32_t *next, *exit;  // claim and exit counters (zero between launches)
};
constexpr int kMaxBatchFields = 1024;

// Item k of the batch: its field (binary search of the positions, read
// through the read-only cache) and record; x = ~0 when none is left.
__device__ __forceinline__ uint4 resolve_batch(const FwdBatch &b, uint32_t k, uint32_t &field) {
    const int n = kCostClasses * b.nfields;
    field = 0;
    if (k >= __ldg(b.pos + n)) return make_uint4(~0u, 0u, 0u, 0u);
    int lo = 0, hi = n - 1;  // largest e with pos[e] <= k
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(b.pos + mid) <= k) lo = mid; else hi = mid - 1;
    }
    field = (uint32_t)(lo % b.nfields);
    return b.args[field].order_rec[__ldg(b.place + lo) + (k - __ldg(b.pos + lo))];
}

// Last block out of a batch launch (one warp): the mean cost of all fields'
// items, and the batch counters reset.
__device__ __forceinline__ void sched_finish_batch(const FwdBatch &b, int lane) {
    int last = 0;
    if (lane == 0) {
        __threadfence();
        last = atomicAdd(b.exit, 1u) == gridDim.x - 1;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    unsigned long long tot = 0ull, items = 0ull;
    for (int f = lane; f < b.nfields; f += 32) {
        tot += __ldcg(b.args[f].sched_total);
        items += (unsigned long long)b.args[f].nitems;
    }
    tot = warp_sum(tot);
    items = warp_sum(items);
    const uint32_t mean = (uint32_t)min(items ? tot / items : 0ull, 0xffffffffull);
    for (int f = lane; f < b.nfields; f += 32) {
        b.args[f].sched[0] = mean;
        *b.args[f].sched_total = 0ull;
    }
    if (lane == 0) {
        *b.next = 0u;
        *b.exit = 0u;
    }
}

// Persistent blocks take work items, heaviest first: block b the b-th, then
// from a global counter (claims past the grid's first items).
// The G warps of a block share an item (equal runs of its candidate list);
// their partial sums are combined in warp order, so Psi does not depend on
// timing.  G = 1 when there are enough items to balance the warps, 2 or 4 for
// small problems.
// ADJ: 0 forward only, 1 with the fused adjoint, 2 with the fused adjoint
// and compensated (Kahan) per-item moment sums.
// BATCH: the items of a batch of fields (b); otherwise of one field (a1).
template <int G, int ADJ, bool BATCH>
__device__ __forceinline__ void forward_loop(const FwdArgs &a1, const FwdBatch &b) {
    // two rings per warp (kernels partly / fully covering the item box); a
    // ring holds 64 staged kernels (32 pairs), consumed 32 at a time from
    // slot 0 or 32
    //
    // Shared memory is kept small: the L1 cache that serves the kernel-record
    // gathers gets what the blocks leave of the SM's unified 256 KB.  A warp's
    // rings are idle during the adjoint, so the nz points live in its first
    // ring and its adjoint queue in the second.
    constexpr int NT = G > 1 ? 2 : kMostTiles;  // tiles of an item (the points of a lane)
    constexpr int GR = G > 1 ? G : 1;    // the cross-warp sums exist only for G > 1
    constexpr int RL = G > 1 ? 32 : 1;
    constexpr int kTouchW = G > 1 ? kTouch / 2 : kTouch;  // kernels remembered per warp
    __shared__ __align__(16) float ringP[G][(kQueue / 2) * kPairFloats];
    __shared__ __align__(16) float ringF[G][(kQueue / 2) * kPairFloats];
    // what the warps of a block exchange, of the current and of the last item
    __shared__ float2 red_psi[2][GR][RL];
    __shared__ uint2 red_n[2][GR][RL];
    __shared__ uint32_t red_cost[2][GR];
    __shared__ uint4 s_rec[2];
    // fused adjoint: the kernels each warp found reaching the item
    __shared__ uint32_t touch[ADJ ? G : 1][ADJ ? kTouchW : 1];
    // batch: the arguments of the current item's field
    __shared__ __align__(16) unsigned char s_args[BATCH ? sizeof(FwdArgs) : 16];
    __shared__ uint32_t s_field[2];
    static_assert(sizeof(NzPoints) <= sizeof(ringP[0]) && kQueue * 4 <= (int)sizeof(ringF[0]), "ring aliases");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    NzPoints &nzs = *reinterpret_cast<NzPoints *>(ringP[warp]);
    uint32_t *adjq = reinterpret_cast<uint32_t *>(ringF[warp]);
    // the first record lies in the slot that the first item does not write: a
    // warp may still have to read it when thread 0 stores the second one
    constexpr int kFirstSlot = 1;
    if (threadIdx.x == 0) {
        if (BATCH) {
            uint32_t f;
            s_rec[kFirstSlot] = resolve_batch(b, blockIdx.x, f);
            s_field[kFirstSlot] = f;
        } else {
            s_rec[kFirstSlot] = resolve(a1, blockIdx.x);
        }
    }
    __syncthreads();
    uint4 rec = s_rec[kFirstSlot];  // the item's record; x = ~0 when done
    uint32_t field = BATCH ? s_field[kFirstSlot] : 0u, loaded = ~0u;
    uint32_t mean = BATCH ? 0u : a1.sched[0];
    const FwdArgs &a = BATCH ? *reinterpret_cast<const FwdArgs *>(s_args) : a1;
    // several warps: buffer of the current item, and the last item's record,
    // whose cost is noted once its warps have met again
    int par = kFirstSlot ^ 1;
    uint4 done = make_uint4(~0u, 0u, 0u, 0u);
    auto note_done = [&]() {
        if (G > 1 && threadIdx.x == 0 && done.x != ~0u) {
            uint32_t c = 0;
#pragma unroll
            for (int q = 0; q < GR; ++q) c += red_cost[par ^ 1][q];
            note_cost(a, mean, done, c);
        }
        done.x = ~0u;
    };
    while (rec.x != ~0u) {
        if (BATCH && field != loaded) {
            // the block's threads copy the field's arguments (block-uniform
            // branch: every thread holds the same record and field)
            if (G == 1) __syncwarp(); else __syncthreads();
            if (loaded != ~0u) note_done();  // with the arguments of its own field
            if (G > 1) __syncthreads();
            const uint32_t *src = reinterpret_cast<const uint32_t *>(b.args + field);
            uint32_t *dst = reinterpret_cast<uint32_t *>(s_args);
            for (int k = threadIdx.x; k < (int)(sizeof(FwdArgs) / 4); k += blockDim.x) dst[k] = src[k];
            if (G == 1) __syncwarp(); else __syncthreads();
            loaded = field;
            mean = a.sched[0];
        }
        const ItemInfo it = item_info(rec);
        // the next claim is made now, its record is fetched after the sums
        // and used at the end, so neither round trip is on the item's path
        uint32_t knext = 0, fnext = 0;
        if (threadIdx.x == 0) knext = gridDim.x + atomicAdd(BATCH ? b.next : a.item_next, 1u);
        f2 acc[NT];
        uint32_t n[NT], cost;
        int ntouch = 0;
        // the targets, for the residuals after the sums: loaded early where
        // registers allow (with one warp per item, or without the adjoint, that
        // cost 1.6 % and 3 %)
        constexpr bool kEarly = G > 1 && ADJ;
        float tv[NT];
        auto targets = [&]() {
#pragma unroll
            for (int p = 0; p < NT; ++p) tv[p] = lane + p * kTile < it.np ? a.t[it.i0 + lane + p * kTile] : 0.f;
        };
        if (kEarly) targets();
        forward_share<G, ADJ>(a, it, warp, ringP[warp], ringF[warp], lane, acc, n, cost, touch[ADJ ? warp : 0], kTouchW,
                              ntouch);
        if (!kEarly) targets();
        uint4 rn = make_uint4(~0u, 0u, 0u, 0u);
        if (threadIdx.x == 0) rn = BATCH ? resolve_batch(b, knext, fnext) : resolve(a, knext);
        if constexpr (G == 1) {
            // one warp: finish the tiles directly
            float ev[NT];
            ff l2 = {0.f, 0.f};
            float mx = 0.f;
            uint32_t cnt = 0u, pr = 0u, pb = 0u, ebits = 0u;
#pragma unroll
            for (int p = 0; p < NT; ++p) {
                float l0, h0, l2p, mxp;
                uint32_t cntp, prp;
                f2_unpack(acc[p], l0, h0);
                ev[p] = point_out(a, it.i0 + lane + p * kTile, lane + p * kTile < it.np, tv[p], l0 + h0, n[p], l2p, mxp,
                                  cntp, prp);
                l2 = ff_add(l2, l2p);
                mx = fmaxf(mx, mxp);
                cnt += cntp;
                pr += prp;
                // adjoint pairs: every support pair of a point with E != 0
                // (the adjoint takes exactly these)
                pb += ev[p] != 0.f ? n[p] : 0u;
                ebits = max(ebits, __float_as_uint(fabsf(ev[p])));
            }
            finish_item(a, it.t0, it.ntl, l2, mx, cnt, pr, lane);
            if (ADJ) ebits = redux_max_u32(ebits);
            if (ADJ && ebits != 0u) {
                pb = redux_add(pb);
                if (lane == 0 && pb) atomicAdd(a.adj_pairs, (unsigned long long)pb);
                float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
                float4 hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
                int nc = 0;
#pragma unroll
                for (int p = 0; p < NT; ++p) {
                    if (p < it.ntl) {
                        const int64_t i = it.i0 + (lane + p * kTile < it.np ? lane + p * kTile : 0);
                        const float x = a.x[i], y = a.y[i], z = a.z[i];
                        nz_grow(lo, hi, ev[p] != 0.f, x, y, z);
                        nc += nz_tile(nzs, nc, ev[p] != 0.f, x, y, z, ev[p], lane);
                    }
                }
                nz_box(lo, hi);
                __syncwarp();
                if ((nc & 1) && lane == 0) nz_pad(nzs, nc);
                __syncwarp();
                adjoint_share<1, (ADJ > 1)>(a, it, 0, nzs, nc, lo, hi, touch[0], ntouch, kTouchW,
                                            __uint_as_float(ebits), adjq, lane, cost);
                __syncwarp();
            }
            if (lane == 0) note_cost(a, mean, rec, cost);
            rec.x = __shfl_sync(0xffffffffu, rn.x, 0);
            rec.y = __shfl_sync(0xffffffffu, rn.y, 0);
            rec.z = __shfl_sync(0xffffffffu, rn.z, 0);
            rec.w = __shfl_sync(0xffffffffu, rn.w, 0);
            if (BATCH) field = __shfl_sync(0xffffffffu, fnext, 0);
            continue;
        } else {
            // the only barrier of an item: the warps' sums, the next record and
            // the last item's costs meet.  Every warp then forms the residuals
            // of both tiles and its own nz points, so none waits for another's;
            // warps 0 and 1 also write a tile each.  (With the nz points made by
            // those two for all there were four barriers, a fifth of the warps'
            // time for 64^3 + 32^3 points.)  A buffer is written again two
            // items later, past the barrier that follows its last reader; the
            // record of the first item lies in the buffer of the second one.
            {
                float l0, h0, l1, h1;
                f2_unpack(acc[0], l0, h0);
                f2_unpack(acc[1], l1, h1);
                red_psi[par][warp][lane] = make_float2(l0 + h0, l1 + h1);
                red_n[par][warp][lane] = make_uint2(n[0], n[1]);
            }
            if (threadIdx.x == 0) {
                s_rec[par] = rn;
                if (BATCH) s_field[par] = fnext;
            }
            __syncthreads();
            note_done();
            float ev[2];
            uint32_t ebits = 0u, pb = 0u;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                float ps = 0.f;
                uint32_t np = 0;
#pragma unroll
                for (int q = 0; q < G; ++q) {
                    const float2 v = red_psi[par][q][lane];
                    const uint2 c = red_n[par][q][lane];
                    ps += t ? v.y : v.x;
                    np += t ? c.y : c.x;
                }
                const bool v = lane + t * kTile < it.np;
                if (warp == t && t < it.ntl) {
                    float l2, mx;
                    uint32_t cnt, pr;
                    ev[t] = point_out(a, it.i0 + lane + t * kTile, v, tv[t], ps, np, l2, mx, cnt, pr);
                    finish_tile(a, it.t0 + t, l2, mx, cnt, pr, lane);
                    // adjoint pairs: every support pair of a point with E != 0
                    pb = ev[t] != 0.f ? np : 0u;
                } else {
                    point_residual(a, v, tv[t], ps, ev[t]);
                }
                ebits = max(ebits, __float_as_uint(fabsf(ev[t])));
            }
            if (ADJ) ebits = redux_max_u32(ebits);
            if (ADJ && ebits != 0u) {
                if (warp < 2) {
                    pb = redux_add(pb);
                    if (lane == 0 && pb) atomicAdd(a.adj_pairs, (unsigned long long)pb);
                }
                float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
                float4 hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
                int nc = 0;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    const int64_t i = it.i0 + (lane + t * kTile < it.np ? lane + t * kTile : 0);
                    const float x = a.x[i], y = a.y[i], z = a.z[i];
                    nz_grow(lo, hi, ev[t] != 0.f, x, y, z);
                    nc += nz_tile(nzs, nc, ev[t] != 0.f, x, y, z, ev[t], lane);
                }
                nz_box(lo, hi);
                __syncwarp();
                if ((nc & 1) && lane == 0) nz_pad(nzs, nc);
                __syncwarp();
                adjoint_share<G, (ADJ > 1)>(a, it, warp, nzs, nc, lo, hi, touch[ADJ ? warp : 0], ntouch,
                                            kTouchW, __uint_as_float(ebits), adjq, lane, cost);
                __syncwarp();
            }
            if (lane == 0) red_cost[par][warp] = cost;
            done = rec;
            rec = s_rec[par];
            if (BATCH) field = s_field[par];
            par ^= 1;
        }
    }
    if (G > 1) {
        __syncthreads();
        note_done();
    }
    // the last block out prepares the next launch: every block has made its
    // last claim and recorded its costs before it counts itself out
    if (BATCH) {
        if (warp == 0) sched_finish_batch(b, lane);
    } else if (threadIdx.x == 0) {
        sched_finish(a1);
    }
}

// Resident warps per SM (the register budget): 16 with one warp per item (four
// points per lane: 126 registers; 20 warps spill 80 bytes and took 2158 us
// instead of 2085 for 9.4 M points), with four, and with two and compensated
// sums (20 spill 116 bytes: 64^3 + 32^3 points 75 us, now 68, 97^3 214 and 193,
// 128^3 374 and 345); 20 for the fused variant with two, 24 with eight (16 spill
// nothing and took 450 us instead of 430 on 128^3) and for the forward alone with
// two or four; measured on the 128^3 and 256^3 fields, other bounds were slower.
#define SERBF_FWD_BOUNDS(G, ADJ) \
    __launch_bounds__(G * 32, (G == 1 ? 16 : (G == 8 ? 24 : (ADJ ? (G == 4 || ADJ == 2 ? 16 : 20) : 24))) / G)

template <int G, int ADJ>
__global__ void SERBF_FWD_BOUNDS(G, ADJ) k_forward(FwdArgs a) {
    pdl_wait();
    pdl_trigger();
    forward_loop<G, ADJ, false>(a, FwdBatch{});
}

// One launch over the work items of every field of a batch.
template <int G, int ADJ>
__global__ void SERBF_FWD_BOUNDS(G, ADJ) k_forward_batch(FwdBatch b) {
    pdl_wait();
    pdl_trigger();
    forward_loop<G, ADJ, true>(FwdArgs{}, b);
}

template <int G, int ADJ>
int launch_forward(const FwdArgs &a, int64_t nitems, int sm_count, cudaStream_t s) {
    static int per_sm = 0;  // resident blocks per SM (same for every device of one kind)
    if (per_sm == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_forward<G, ADJ>, G * 32, 0) != cudaSuccess ||
            nb < 1)
            return SERBF_ECUDA;
        per_sm = nb;
    }
    int64_t blocks = nitems;
    const int64_t resident = (int64_t)sm_count * per_sm;
    if (blocks > resident) blocks = resident;
    launch_pdl(k_forward<G, ADJ>, dim3((unsigned)blocks), dim3(G * 32), 0, s, a);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

// After the forward: the Eq. 3-19 loss terms from the tile partials in tile
// order (a warp per group of kFwdGroup tiles, then the last block over the
// group partials), and with the fused adjoint the ten App. A gradients of each
// kernel from its fixed-point moments (a thread per kernel, accumulators
// cleared for the next launch).  The last block writes the totals.
constexpr float kFixUnitF = 1.4551915228366852e-11f;  // 2^-36
constexpr int kFinishThreads = 256;

struct FinishArgs {
    const FwdPart *part;
    FwdGPart *gpart;
    int64_t ntiles;
    const float *p;
    const int32_t *m_dev;
    int cap;
    unsigned long long *fix, *pairs;
    float *grad;
    uint32_t *counter;
    double *stats;
    const float4 *kbwd;      // (c, r2) of each kernel
    float cell_h;            // binning cell edge
    uint32_t *cell_max;      // [0] most points in one cell, [1] running range bound (float bits)
    const float4 *field_box; // box of all binned points
    float npoints;
    int32_t *status;
};

// Upper bound of |moment| / max|E| for kernel j (centre c, support radius
// r): a pair has phi <= 1 and every component of v - c is at most the
// distance from c to the farthest corner of the points' box, and below r,
// so every moment of the kernel is at most (points within r of c) * max|E| *
// max(1, min(r^2, far^2)); the points within r are at most the points of
// the field and at most (cells a ball of radius r can touch) * (most points
// in one cell).
__device__ __forceinline__ float moment_bound(float4 k0, float h, uint32_t cell_max, const float4 *box, float npts) {
    const float nc = ceilf(2.f * sqrtf(k0.w) / h) + 2.f;
    const float far2 = box_far_d2(k0.x, k0.y, k0.z, box[0], box[1]);
    return fmaxf(1.f, fminf(k0.w, far2)) * fminf(npts, nc * nc * nc * (float)cell_max);
}

// Block bx of nbx.
template <bool ADJ>
__device__ __forceinline__ void fwd_finish_body(const FinishArgs &f, int bx, int nbx) {
    __shared__ bool s_last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t ngroups = (f.ntiles + kFwdGroup - 1) / kFwdGroup;
    const int64_t g = (int64_t)bx * (kFinishThreads / 32) + warp;
    if (g < ngroups) {
        const uint32_t gb = (uint32_t)(g * kFwdGroup);
        const uint32_t ge = (uint32_t)min((int64_t)gb + kFwdGroup, f.ntiles);
        const FwdGPart gp = reduce_parts(f.part, gb, ge, lane);
        if (lane == 0) f.gpart[g] = gp;
    }
    if (ADJ) {
        const int m = *f.m_dev;
        const int j = bx * blockDim.x + threadIdx.x;
        if (j < m) {
            unsigned long long *o = f.fix + 10 * (size_t)j;
            float M[10];
#pragma unroll
            for (int r = 0; r < 10; ++r) {
                // int64 -> float from its two 32-bit halves and one FMA;
                // relative error ~1e-7
                const long long v = (long long)o[r];
                const float hi = (float)(int)(v >> 32), lo = (float)(uint32_t)(v & 0xffffffffll);
                M[r] = fmaf(hi, 4294967296.f, lo) * kFixUnitF;
                o[r] = 0ull;
            }
            grad_from_moments<true>(f.p, f.cap, j, M, f.grad);
            // positive floats order like their bits (NaN orders above +inf)
            atomicMax(&f.cell_max[1], __float_as_uint(moment_bound(f.kbwd[4 * j], f.cell_h, f.cell_max[0],
                                                                   f.field_box, f.npoints)));
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(f.counter, 1u) == (unsigned)nbx - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // every warp of the last block takes an equal run of the groups, the first
    // one then their sums (one warp over all groups took half of the launch's
    // 33 us for 9.4 M points, which now takes 17)
    __shared__ FwdGPart s_part[kFinishThreads / 32];
    constexpr int NW = kFinishThreads / 32;
    const uint32_t per = (uint32_t)((ngroups + NW - 1) / NW);
    const uint32_t b0 = min(per * warp, (uint32_t)ngroups), b1 = min(per * (warp + 1), (uint32_t)ngroups);
    const FwdGPart own = reduce_parts(f.gpart, b0, b1, lane);
    if (lane == 0) s_part[warp] = own;
    __syncthreads();
    if (warp != 0) return;
    if (lane == 0) {
        FwdGPart tot = s_part[0];
#pragma unroll
        for (int w = 1; w < NW; ++w) {
            tot.l2 += s_part[w].l2;
            tot.maxe = fmaxf(tot.maxe, s_part[w].maxe);
            tot.cnt += s_part[w].cnt;
            tot.pairs += s_part[w].pairs;
        }
        f.stats[SERBF_STAT_L2] = tot.l2;
        f.stats[SERBF_STAT_MAXE] = tot.maxe;
        f.stats[SERBF_STAT_COUNT] = (double)tot.cnt;
        f.stats[SERBF_STAT_PAIRS_FWD] = (double)tot.pairs;
        if (ADJ) {
            f.stats[SERBF_STAT_PAIRS_BWD] = (double)__ldcg(f.pairs);
            *f.pairs = 0ull;
            // the int64 sums hold |moment| < 2^27 (unit 2^-36); flag when the
            // bound reaches 2^26, or is not finite
            const float bound = __uint_as_float(__ldcg(&f.cell_max[1])) * tot.maxe;
            if (!(bound < 67108864.f)) atomicOr(f.status, SERBF_FLAG_FIX_RANGE);
            f.cell_max[1] = 0u;
        }
        *f.counter = 0u;
    }
}

template <bool ADJ>
__global__ void __launch_bounds__(kFinishThreads) k_fwd_finish(FinishArgs f) {
    pdl_wait();
    pdl_trigger();
    fwd_finish_body<ADJ>(f, blockIdx.x, gridDim.x);
}

// Batch: field blockIdx.y.
template <bool ADJ>
__global__ void __launch_bounds__(kFinishThreads) k_fwd_finish_batch(const FinishArgs *fa) {
    pdl_wait();
    pdl_trigger();
    const FinishArgs f = fa[blockIdx.y];
    fwd_finish_body<ADJ>(f, blockIdx.x, gridDim.x);
}

// The arguments of one forward (+ adjoint) call with G warps per item; false
// on bad arguments.
bool make_args(const serbf_points *pts, const serbf_params *prm, const serbf_config *cfg, float *psi, float *err,
               uint8_t *mask, float *grad, double *stats, serbf_workspace *ws, int G, FwdArgs &a, FinishArgs &f,
               int64_t &finish_blocks) {
    if (!pts || !prm || !cfg || !ws || ws->magic != kMagic || !ws->binned) return false;
    if (pts->n != ws->npoints || !prm->m || !prm->p) return false;
    if (pts->n > 0 && (!pts->x || !pts->y || !pts->z || !pts->t || !psi || !err || !mask)) return false;
    if (!stats) return false;
    const bool adj = grad != nullptr;
    if (cfg->fwd_warps != 0 && cfg->fwd_warps != 1 && cfg->fwd_warps != 2 && cfg->fwd_warps != 4 && cfg->fwd_warps != 8)
        return false;
    if (adj && (prm->cap < 1 || prm->cap > ws->sz.max_kernels)) return false;
    a.x = pts->x;
    a.y = pts->y;
    a.z = pts->z;
    a.t = pts->t;
    const ItemSet &items = items_of(ws, G);
    a.order_rec = items.order;
    a.item_class = items.cls;
    a.sched = items.sched;
    a.sched_total = items.total;
    a.nitems = items.n;
    a.tile_lo = ws->tile_lo;
    a.tile_hi = ws->tile_hi;
    a.slist = ws->sup_list;
    a.scnt = ws->sup_cnt;
    a.kfwd = ws->kfwd;
    a.adj_fix = ws->adj_fix;
    a.adj_pairs = ws->adj_pairs;
    a.scap = ws->sz.super_cap;
    // float thresholds that give the same decisions as comparing in double:
    // t <= tau1 iff t <= (largest float <= tau1), t >= tau2 iff t >= (smallest float >= tau2)
    a.tau1 = (float)cfg->tau1;
    if ((double)a.tau1 > cfg->tau1) a.tau1 = nextafterf(a.tau1, -INFINITY);
    a.tau2 = (float)cfg->tau2;
    if ((double)a.tau2 < cfg->tau2) a.tau2 = nextafterf(a.tau2, INFINITY);
    a.psi = psi;
    a.err = err;
    a.mask = mask;
    a.part = ws->fwd_part;
    a.item_next = ws->counters + 4;
    a.exit_count = ws->counters + 6;
    a.status = ws->status;
    f.part = ws->fwd_part;
    f.gpart = reinterpret_cast<FwdGPart *>(ws->fwd_gpart);
    f.ntiles = ws->ntiles;
    f.p = prm->p;
    f.m_dev = prm->m;
    f.cap = prm->cap;
    f.fix = ws->adj_fix;
    f.pairs = ws->adj_pairs;
    f.grad = grad;
    f.counter = ws->counters + 5;
    f.stats = stats;
    f.kbwd = ws->kbwd;
    f.cell_h = ws->grid.h;
    f.cell_max = ws->cell_max;
    f.field_box = ws->field_box;
    f.npoints = (float)ws->npoints;
    f.status = ws->status;
    const int64_t ngroups = (ws->ntiles + kFwdGroup - 1) / kFwdGroup;
    int64_t nb = (ngroups + kFinishThreads / 32 - 1) / (kFinishThreads / 32);
    if (adj) nb = max(nb, (int64_t)((prm->cap + kFinishThreads - 1) / kFinishThreads));
    finish_blocks = nb < 1 ? 1 : nb;
    return true;
}

int forward_impl(const serbf_points *pts, const serbf_params *prm, const serbf_config *cfg, float *psi, float *err,
                 uint8_t *mask, float *grad, double *stats, serbf_workspace *ws, void *stream) {
    FwdArgs a;
    FinishArgs f;
    int64_t nb = 1;
    if (!cfg || !ws || ws->magic != kMagic) return SERBF_EINVAL;
    const int G = forward_warps(ws->items[1].n, ws->sm_count, cfg->fwd_warps);
    if (!make_args(pts, prm, cfg, psi, err, mask, grad, stats, ws, G, a, f, nb)) return SERBF_EINVAL;
    const bool adj = grad != nullptr;
    cudaStream_t s = (cudaStream_t)stream;
    int rc = SERBF_OK;
    if (ws->ntiles > 0) {
        ws->unmeasured = 0;
        const int64_t ni = a.nitems;
        const int mode = adj ? (cfg->kahan ? 2 : 1) : 0;
        switch (G * 4 + mode) {
            case 4: rc = launch_forward<1, 0>(a, ni, ws->sm_count, s); break;
            case 5: rc = launch_forward<1, 1>(a, ni, ws->sm_count, s); break;
            case 6: rc = launch_forward<1, 2>(a, ni, ws->sm_count, s); break;
            case 8: rc = launch_forward<2, 0>(a, ni, ws->sm_count, s); break;
            case 9: rc = launch_forward<2, 1>(a, ni, ws->sm_count, s); break;
            case 10: rc = launch_forward<2, 2>(a, ni, ws->sm_count, s); break;
            case 16: rc = launch_forward<4, 0>(a, ni, ws->sm_count, s); break;
            case 17: rc = launch_forward<4, 1>(a, ni, ws->sm_count, s); break;
            case 18: rc = launch_forward<4, 2>(a, ni, ws->sm_count, s); break;
            case 32: rc = launch_forward<8, 0>(a, ni, ws->sm_count, s); break;
            case 33: rc = launch_forward<8, 1>(a, ni, ws->sm_count, s); break;
            default: rc = launch_forward<8, 2>(a, ni, ws->sm_count, s); break;
        }
    }
    if (rc) return rc;
    if (adj)
        launch_pdl(k_fwd_finish<true>, dim3((unsigned)nb), dim3(kFinishThreads), 0, s, f);
    else
        launch_pdl(k_fwd_finish<false>, dim3((unsigned)nb), dim3(kFinishThreads), 0, s, f);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

template <int G, int ADJ>
int launch_forward_batch(const FwdBatch &b, int64_t nitems, int sm_count, cudaStream_t s) {
    static int per_sm = 0;
    if (per_sm == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_forward_batch<G, ADJ>, G * 32, 0) != cudaSuccess ||
            nb < 1)
            return SERBF_ECUDA;
        per_sm = nb;
    }
    int64_t blocks = nitems;
    const int64_t resident = (int64_t)sm_count * per_sm;
    if (blocks > resident) blocks = resident;
    if (blocks < 1) blocks = 1;
    launch_pdl(k_forward_batch<G, ADJ>, dim3((unsigned)blocks), dim3(G * 32), 0, s, b);
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

}  // namespace

namespace serbf {

size_t fwd_args_size() { return sizeof(FwdArgs); }
size_t finish_args_size() { return sizeof(FinishArgs); }

// Host records of one field's fused forward + adjoint (out: sizeof(FwdArgs)
// and sizeof(FinishArgs) bytes) and the finishing kernel's block count.
int batch_forward_args(const serbf_points *pts, const serbf_params *prm, const serbf_config *cfg, float *psi,
                       float *err, uint8_t *mask, float *grad, double *stats, serbf_workspace *ws, int G, void *fwd_out,
                       void *fin_out, int64_t *finish_blocks) {
    FwdArgs a;
    FinishArgs f;
    if (!make_args(pts, prm, cfg, psi, err, mask, grad, stats, ws, G, a, f, *finish_blocks)) return SERBF_EINVAL;
    memcpy(fwd_out, &a, sizeof(a));
    memcpy(fin_out, &f, sizeof(f));
    return SERBF_OK;
}

// One persistent launch over the items of every field, then the finishing
// kernel of every field (grid.y = field).  args / fin / counters are device
// arrays written by the batch set-up, table by the batched rebuild.
int batch_forward_launch(const void *args, const void *fin, const uint32_t *table, int nfields, uint32_t *counters,
                         int64_t total_items, int64_t finish_blocks, int G, int kahan, int sm_count, cudaStream_t s) {
    if (nfields < 1 || nfields > kMaxBatchFields) return SERBF_EINVAL;
    FwdBatch b{static_cast<const FwdArgs *>(args), table, table + kCostClasses * nfields + 1, nfields, counters, counters + 1};
    int rc = SERBF_OK;
    if (total_items > 0) {
        switch (G * 2 + (kahan ? 1 : 0)) {
            case 2: rc = launch_forward_batch<1, 1>(b, total_items, sm_count, s); break;
            case 3: rc = launch_forward_batch<1, 2>(b, total_items, sm_count, s); break;
            case 4: rc = launch_forward_batch<2, 1>(b, total_items, sm_count, s); break;
            case 5: rc = launch_forward_batch<2, 2>(b, total_items, sm_count, s); break;
            case 8: rc = launch_forward_batch<4, 1>(b, total_items, sm_count, s); break;
            case 9: rc = launch_forward_batch<4, 2>(b, total_items, sm_count, s); break;
            case 16: rc = launch_forward_batch<8, 1>(b, total_items, sm_count, s); break;
            case 17: rc = launch_forward_batch<8, 2>(b, total_items, sm_count, s); break;
            default: return SERBF_EINVAL;
        }
    }
    if (rc) return rc;
    launch_pdl(k_fwd_finish_batch<true>, dim3((unsigned)finish_blocks, (unsigned)nfields), dim3(kFinishThreads), 0, s,
               static_cast<const FinishArgs *>(fin));
    SERBF_CHECK_LAUNCH();
    return SERBF_OK;
}

}  // namespace serbf

extern "C" int serbf_forward(const serbf_points *pts, const serbf_params *prm, const serbf_config *cfg, float *psi,
                             float *err, uint8_t *mask, double *stats, serbf_workspace *ws, void *stream) {
    SERBF_TRACE();
    return forward_impl(pts, prm, cfg, psi, err, mask, nullptr, stats, ws, stream);
}

extern "C" int serbf_forward_backward(const serbf_points *pts, const serbf_params *prm, const serbf_config *cfg,
                                      float *psi, float *err, uint8_t *mask, float *grad, double *stats,
                                      serbf_workspace *ws, void *stream) {
    SERBF_TRACE();
    if (!grad) return SERBF_EINVAL;
    return forward_impl(pts, prm, cfg, psi, err, mask, grad, stats, ws, stream);
}
