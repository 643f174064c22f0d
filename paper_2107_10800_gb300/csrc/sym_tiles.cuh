// Symmetric products on 32 x 32 warp tiles: u = N g for a symmetric pair
// tensor N (N_ji = N_ij^T), each unordered pair evaluated once and applied in
// both directions.  The pair's arithmetic is a policy: FP64 here and in
// single_blob.cu, double-float in rpy_df.cu; a tile's sums are in that
// arithmetic, the sums over tiles in FP64.
//
// A warp takes a tile of 32 targets, one per lane, against 32 sources staged
// in its own shared memory: at step t lane l meets source (l + t) mod 32, the
// target's sum stays on the lane and the source's column sum moves one lane
// per step, so that it meets every target once.  On a tile against itself
// steps 1..15, and 16 on half the lanes, take every unordered pair once (step
// 0: the self term).  A work item is a pair of groups of whole tiles (I <= J)
// of one system; its warp walks the tile pairs, keeps a target tile's sums in
// registers across the source tiles and adds the column sums to the item's
// own slots of the partial sums, so the order of every sum is fixed and the
// result does not depend on scheduling.  The slots (one per group of the
// system) are added by the caller.
//
// Why this shape: GB300 issues 2 FP64 multiply-adds per SM and cycle (16
// cycles for a warp), so the FP64 pipe bounds the product and nothing but FP64
// operations counts; a warp that needs no block barrier and stages its own
// sources keeps the pipe fed with 4 to 5 warps per scheduler.  Groups of
// several tiles (up to 96 groups per system) bound the partial sums at 96
// slots; systems too small to give every SM a few warps split the 32 steps
// of a tile over up to 8 items (each with its own slots).  Measured against
// the block-wide form it replaced (four warps or one, shared-memory sums of
// every warp tile): 384 free blobs 108 -> 15 us (78 unsplit tiles keep 78 SMs
// busy with 14 us of FP64 issue each), 2,560 wall blobs 533 -> 508 us, 5,000
// wall blobs 1,851 -> 1,885 us.
#pragma once
#include "am_internal.cuh"
#include "rpy_pair.cuh"

#include <algorithm>
#include <type_traits>
#include <vector>

namespace am {

// One warp per block: the blocks of a launch then spread evenly over the SMs
// whatever their number (2,560 blobs make 3,240 items, 21.3 per SM).  An SM holds
// 25 of them above a wall (78 registers) and 21 in free space (95): such a
// launch is one wave, or one and a few items.
constexpr int kSymWarps = 1;
constexpr int kSymMaxGroups = 96;  // most groups (partial-sum slots) per system
// the same for the paired-lane product, whose items run one per block of four
// warps: about 12,000 items keep the last wave of a large product short
constexpr int kPairMaxGroups = 160;

// Values of the FP64 policies.
struct SymFp64 {
    using V = double;
    static __device__ __forceinline__ double ld(double x) { return x; }
    static __device__ __forceinline__ double to(double x) { return x; }
    static __device__ __forceinline__ double shfl(double x, int lane) { return __shfl_sync(0xffffffffu, x, lane); }
};

// The blob mobility (3 components), free space or wall; sums in units of A1.
template <bool WALL>
struct SymBlobPair : SymFp64 {
    static constexpr int NC = 3;
    static constexpr int kMinBlocks = WALL ? 22 : 20;  // 78 and 95 registers, no spills
    RpyK<double> k;
    explicit SymBlobPair(const RpyK<double>& q) : k(q) {}
    __device__ __forceinline__ double scale() const { return k.A1; }
    __device__ __forceinline__ void both(const double* xi, const double* xj, const double* l, const double* m,
                                         double* u, double* v) const {
        const double dx = xi[0] - xj[0], dy = xi[1] - xj[1], dz = xi[2] - xj[2];
        if (WALL) {
            const double rxy2 = fma(dx, dx, dy * dy);
            pair_wall_sym<double>(dx, dy, dz, rxy2, fma(dz, dz, rxy2), xi[2] + xj[2], 2.0 * xj[2], -xi[2], l[0], l[1],
                                  l[2], m[0], m[1], m[2], k, u[0], u[1], u[2], v[0], v[1], v[2]);
        } else {
            pair_free_sym<double>(dx, dy, dz, fma(dx, dx, fma(dy, dy, dz * dz)), l[0], l[1], l[2], m[0], m[1], m[2], k,
                                  u[0], u[1], u[2], v[0], v[1], v[2]);
        }
    }
    __device__ __forceinline__ void self(const double* xi, const double* m, double* u) const {
        if (WALL)
            pair_wall_r2<double>(0.0, 0.0, 0.0, 0.0, 0.0, 2.0 * xi[2], 2.0 * xi[2], -xi[2], m[0], m[1], m[2], k, u[0],
                                 u[1], u[2]);
        else
            pair_free<double>(0.0, 0.0, 0.0, m[0], m[1], m[2], k, u[0], u[1], u[2]);
    }
};

// The items of one system of n without a list: groups of T, ng of them, the
// steps split `splits` ways (items as sym_append_items makes them, poff = 0).
struct SymSpan {
    int n = 0, T = 32, ng = 0, splits = 1;
};

__device__ __forceinline__ SymItem sym_span_item(const SymSpan& sp, int nc, int idx) {
    const int k = idx % sp.splits, p = idx / sp.splits;
    // row a of the upper triangle starts at a ng - a (a - 1) / 2
    const float w = 2.f * sp.ng + 1.f;
    int a = (int)((w - sqrtf(fmaxf(0.f, w * w - 8.f * p))) * 0.5f);
    a = max(0, min(a, sp.ng - 1));
    while (a > 0 && a * sp.ng - a * (a - 1) / 2 > p) --a;
    while ((a + 1) * sp.ng - (a + 1) * a / 2 <= p) ++a;
    const int b = a + p - (a * sp.ng - a * (a - 1) / 2);
    SymItem m;
    m.i0 = a * sp.T; m.ni = min(sp.T, sp.n - m.i0);
    m.j0 = b * sp.T; m.nj = min(sp.T, sp.n - m.j0);
    m.tbase = 0; m.sys = 0;
    m.ti = a * sp.splits + k; m.tj = b * sp.splits + k;
    m.poff = 0; m.n3 = nc * sp.n;
    m.steps = (32 * k / sp.splits) | (32 * (k + 1) / sp.splits) << 8;
    return m;
}

// x: positions, g: NC values per target, both indexed by the items' blob (or
// body) numbers; part: the slots.  counter[0]: next item, counter[1]: blocks
// finished (NULL: warp w takes items w, w + warps, ..).  items NULL: those of
// `span`.
template <class Pair>
__global__ void __launch_bounds__(32 * kSymWarps, Pair::kMinBlocks)
k_sym_tiles(const double* __restrict__ x, const double* __restrict__ g, double* __restrict__ part,
            const SymItem* __restrict__ items, int n_items, int* __restrict__ counter, Pair pr,
            const int* __restrict__ active, SymSpan span) {
    dep_wait();
    using V = typename Pair::V;
    constexpr int NC = Pair::NC;
    constexpr bool kFp64 = std::is_same_v<V, double>;
    __shared__ V sx[kSymWarps][3 + NC][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    V(*src)[32] = sx[warp];
    const int warps = (int)gridDim.x * kSymWarps;
    for (int round = 0;; ++round) {
        int itn = blockIdx.x + warp * gridDim.x + round * warps;  // the first items spread over the SMs
        if (counter && round > 0) {  // taken only when the warp is free: no item waits for a busy one
            if (lane == 0) itn = warps + atomicAdd(counter, 1);
            itn = __shfl_sync(0xffffffffu, itn, 0);
        }
        if (itn >= n_items) break;
        const SymItem m = items ? items[itn] : sym_span_item(span, NC, itn);
        const bool diag = m.ti == m.tj;
        double* rowo = part + m.poff + (long long)m.tj * m.n3 + NC * (long long)(m.i0 - m.tbase);
        double* colo = part + m.poff + (long long)m.ti * m.n3 + NC * (long long)(m.j0 - m.tbase);
        if (active && !active[m.sys]) {  // a stopped system: zero partial sums
            for (int q = lane; q < NC * m.ni; q += 32) rowo[q] = 0.0;
            if (!diag)
                for (int q = lane; q < NC * m.nj; q += 32) colo[q] = 0.0;
            continue;
        }
        const int s0 = m.step0(), s1 = m.step1();
        const double scale = pr.scale();
        for (int ia = 0; ia < m.ni; ia += 32) {
            const int t = ia + lane;
            const bool ti_ok = t < m.ni;
            V xi[3], mu[NC], u[NC];
            double U[NC];  // sums over tiles (FP64 policies keep them in u)
#pragma unroll
            for (int c = 0; c < 3; ++c) xi[c] = Pair::ld(ti_ok ? x[3 * (size_t)(m.i0 + t) + c] : 1.0);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                mu[c] = Pair::ld(ti_ok ? g[NC * (size_t)(m.i0 + t) + c] : 0.0);
                u[c] = Pair::ld(0.0);
                U[c] = 0.0;
            }
            for (int jb = diag ? ia : 0; jb < m.nj; jb += 32) {
                const bool self_tile = diag && jb == ia;
                __syncwarp();
                {
                    const int q = jb + lane;
                    const bool ok = q < m.nj;
#pragma unroll
                    for (int c = 0; c < 3; ++c) src[c][lane] = Pair::ld(ok ? x[3 * (size_t)(m.j0 + q) + c] : 1.0);
#pragma unroll
                    for (int c = 0; c < NC; ++c) src[3 + c][lane] = Pair::ld(ok ? g[NC * (size_t)(m.j0 + q) + c] : 0.0);
                }
                __syncwarp();
                V v[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    v[c] = Pair::ld(0.0);
                    if (!kFp64) u[c] = Pair::ld(0.0);
                }
#pragma unroll 1
                for (int step = s0; step < s1; ++step) {
                    const int q = (lane + step) & 31;
                    const bool ok = ti_ok && jb + q < m.nj &&
                                    (!self_tile || (step >= 1 && (step < 16 || (step == 16 && lane < 16))));
                    if (ok) {
                        V xj[3], l[NC];
#pragma unroll
                        for (int c = 0; c < 3; ++c) xj[c] = src[c][q];
#pragma unroll
                        for (int c = 0; c < NC; ++c) l[c] = src[3 + c][q];
                        pr.both(xi, xj, l, mu, u, v);
                    } else if (self_tile && step == 0 && ti_ok) {
                        pr.self(xi, mu, u);
                    }
                    // hand the column sum to the lane that meets this source next
#pragma unroll
                    for (int c = 0; c < NC; ++c) v[c] = Pair::shfl(v[c], (lane + 1) & 31);
                }
                // lane l now holds the column sum of source (l + s1) mod 32
                if (self_tile) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const V t = Pair::shfl(v[c], (lane - s1) & 31);
                        if constexpr (kFp64) u[c] += t; else U[c] += Pair::to(t);
                    }
                } else {
                    const int q = jb + ((lane + s1) & 31);
                    if (q < m.nj) {
                        double* o = colo + NC * (size_t)q;
#pragma unroll
                        for (int c = 0; c < NC; ++c)
                            o[c] = ia == 0 ? scale * Pair::to(v[c]) : fma(scale, Pair::to(v[c]), o[c]);
                    }
                }
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (!kFp64) U[c] += Pair::to(u[c]);
            }
            // the rows of a diagonal item also hold the column sums of its
            // earlier target tiles
            __syncwarp();
            if (ti_ok) {
                double* o = rowo + NC * (size_t)t;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const double a = kFp64 ? Pair::to(u[c]) : U[c];
                    o[c] = diag && ia > 0 ? fma(scale, a, o[c]) : scale * a;
                }
            }
        }
    }
    if (counter) item_queue_done(counter);
}

// Tiles per group of a system of n: at most kSymMaxGroups groups.
inline int sym_group_tiles(int n) {
    const int tiles = (n + 31) / 32;
    return tiles <= kSymMaxGroups ? 1 : (tiles + kSymMaxGroups - 1) / kSymMaxGroups;
}

// Splits of a tile's 32 steps (1, 2, 4 or 8) so that `items` items give the
// GPU about two warps per scheduler (8 per SM).
inline int sym_step_splits(long long items) {
    int sp = 1;
    while (sp < 8 && items * sp * 2 <= 8LL * num_sms()) sp *= 2;
    return sp;
}

// Appends the items of one system: blobs base .. base + n - 1 in groups of
// 32 `tiles`, steps split `splits` ways, partial sums at poff in slots of nc n
// doubles.  Returns the number of slots.
inline int sym_append_items(std::vector<SymItem>& out, int sys, int base, int n, int nc, int tiles, int splits,
                            long long poff) {
    const int T = 32 * tiles, ng = (n + T - 1) / T;
    for (int a = 0; a < ng; ++a)
        for (int b = a; b < ng; ++b)
            for (int k = 0; k < splits; ++k) {
                SymItem it;
                it.i0 = base + a * T; it.ni = std::min(T, n - a * T);
                it.j0 = base + b * T; it.nj = std::min(T, n - b * T);
                it.tbase = base; it.sys = sys;
                it.ti = a * splits + k; it.tj = b * splits + k;
                it.poff = poff; it.n3 = nc * n;
                it.steps = (32 * k / splits) | (32 * (k + 1) / splits) << 8;
                out.push_back(it);
            }
    return ng * splits;
}

}  // namespace am
