// One-direction blob mobility product of a range of targets: u = M lambda on
// thread-block clusters in a single launch, or, for more work, on single CTAs
// with slots for parts of the sources.
//
// A cluster takes a group of G targets (G = 8, 16 or 32) and splits the
// sources over its CTAs (at most 8); in a CTA of 128 threads thread t holds
// target t mod G and meets every (128 / G)-th source of the CTA's share from
// t / G on, staged in shared memory 128 at a time.  The 128 / G sums of a
// target are added in the CTA, the CTAs' sums by the first one through
// distributed shared memory, both in a fixed order.  With several parts every
// cluster takes one part of the sources and writes the part's slot (3 nt
// doubles); the slots are added afterwards.
//
// What bounds it and why this split: 384 free blobs are 147,456 pairs of 28
// FP64 operations, 6.4 us if all 152 SMs work (2 FP64 multiply-adds per SM
// and cycle); blocks of 128 targets and 128 sources gave 200 blobs to 4 SMs
// (172 us with its three launches; here 8.0 us).  G, the cluster size and the
// parts are chosen by the expected time (small_shape); positions are read as
// they are, so a small product needs no packing launch, no workspace and no
// second launch for the sums.  The row ranges of a sharded suspension take it
// at every size: 5,003 rows of 20,011 free blobs FP64 6.28 -> 5.04 ms, 949 rows
// of 7,594 wall blobs FP64 1.27 -> 0.96 ms, mixed 54 -> 40 us.
//
// FP32 pair terms (T = float) as in rpy_items_mixed: differences from the hi
// parts, lo parts added within a quarter of the target's largest coordinate;
// FP32 sums over blocks of 16 consecutive sources (16 b .. 16 b + 15 of the
// suspension, in order), added to compensated (hi, lo) sums.  The blocks are
// the same whatever the shape of the launch, so the result depends on it by
// the last bits of a 48-bit sum only.
#pragma once
#include "am_internal.cuh"
#include "dev_util.cuh"
#include "rpy_pair.cuh"
#include "rpy_pair2.cuh"

#include <algorithm>
#include <cmath>

namespace am {

// sources per FP32 partial sum of the mixed kernels before it is added to
// the tile's compensated (hi, lo) sums
constexpr int kSumBlock = 16;

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned v;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(v));
    return v;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned v;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(v));
    return v;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the double at `p` (this CTA's shared memory) in CTA `rank` of the cluster
__device__ __forceinline__ double cluster_load(const double* p, unsigned rank) {
    unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p)), b;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(a), "r"(rank));
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(b) : "memory");
    return v;
}

constexpr int kSmallThreads = 128;
constexpr int kSmallTile = 128;  // sources staged at a time

template <class T>
struct SmallTile;
template <>
struct SmallTile<double> {
    double x[kSmallTile], y[kSmallTile], z[kSmallTile], lx[kSmallTile], ly[kSmallTile], lz[kSmallTile];
};
template <>
struct SmallTile<float> {
    // one entry of padding per block of 16: a warp's threads may be in
    // different blocks
    static constexpr int kSize = kSmallTile + kSmallTile / kSumBlock;
    static __device__ __forceinline__ int at(int q) { return q + q / kSumBlock; }
    float4 h[kSize], o[kSize], l[kSize];  // hi (w: twice the height), lo, forces
};

// Targets t0 .. t0 + nt - 1 against sources 0 .. n - 1; u: 3 nt doubles.
template <class T, bool WALL, int G>
__global__ void __launch_bounds__(kSmallThreads)
k_rpy_small(const double* __restrict__ r, const double* __restrict__ lam, double* __restrict__ u, int n, int t0,
            int nt, int parts, RpyK<T> k) {
    dep_wait();
    constexpr int NS = kSmallThreads / G;
    __shared__ SmallTile<T> tile;
    __shared__ double red[NS][3][G];
    __shared__ double own[3 * G];
    const int rank = (int)cluster_rank(), cs = (int)cluster_size();
    const int group = blockIdx.x / cs / parts, part = blockIdx.x / cs % parts;
    const int e = threadIdx.x % G, sub = threadIdx.x / G;
    const int it = group * G + e;  // target within the rows
    // whole blocks of kSumBlock sources per CTA
    const int nb = (n + kSumBlock - 1) / kSumBlock;
    const int piece = part * cs + rank, pieces = parts * cs;
    const int j0 = kSumBlock * (int)((long long)nb * piece / pieces);
    const int j1 = min(n, kSumBlock * (int)((long long)nb * (piece + 1) / pieces));
    u += (size_t)part * 3 * nt;
    double x = 0.0, y = 0.0, z = 1.0;
    if (it < nt) {
        const double* p = r + 3 * (size_t)(t0 + it);
        x = p[0]; y = p[1]; z = p[2];
    }
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    if constexpr (sizeof(T) == 8) {
        for (int jt = j0; jt < j1; jt += kSmallTile) {
            const int cnt = min(kSmallTile, j1 - jt);
            __syncthreads();
            if ((int)threadIdx.x < cnt) {
                const double* p = r + 3 * (size_t)(jt + threadIdx.x);
                const double* f = lam + 3 * (size_t)(jt + threadIdx.x);
                tile.x[threadIdx.x] = p[0]; tile.y[threadIdx.x] = p[1]; tile.z[threadIdx.x] = p[2];
                tile.lx[threadIdx.x] = f[0]; tile.ly[threadIdx.x] = f[1]; tile.lz[threadIdx.x] = f[2];
            }
            __syncthreads();
#pragma unroll 2
            for (int q = sub; q < cnt; q += NS) {
                const double dx = x - tile.x[q], dy = y - tile.y[q], zj = tile.z[q], dz = z - zj;
                if (WALL) {
                    const double rxy2 = fma(dx, dx, dy * dy);
                    pair_wall_r2<double>(dx, dy, dz, rxy2, fma(dz, dz, rxy2), z + zj, 2.0 * zj, -z, tile.lx[q],
                                         tile.ly[q], tile.lz[q], k, s0, s1, s2);
                } else {
                    pair_free<double>(dx, dy, dz, tile.lx[q], tile.ly[q], tile.lz[q], k, s0, s1, s2);
                }
            }
        }
    } else {
        const float hx = (float)x, hy = (float)y, hz = (float)z;
        const float ox = (float)(x - hx), oy = (float)(y - hy), oz = (float)(z - hz);
        const float nr = 0.25f * fmaxf(fabsf(hx), fmaxf(fabsf(hy), fabsf(hz)));
        const float near2 = nr * nr;
        float th[3] = {0.f, 0.f, 0.f}, tl[3] = {0.f, 0.f, 0.f};
        for (int jt = j0; jt < j1; jt += kSmallTile) {
            const int cnt = min(kSmallTile, j1 - jt);
            __syncthreads();
            if ((int)threadIdx.x < cnt) {
                const double* p = r + 3 * (size_t)(jt + threadIdx.x);
                const double* f = lam + 3 * (size_t)(jt + threadIdx.x);
                const double px = p[0], py = p[1], pz = p[2];
                const float ax = (float)px, ay = (float)py, az = (float)pz;
                const int e2 = tile.at(threadIdx.x);
                tile.h[e2] = make_float4(ax, ay, az, 2.f * az);
                tile.o[e2] = make_float4((float)(px - ax), (float)(py - ay), (float)(pz - az), 0.f);
                tile.l[e2] = make_float4((float)f[0], (float)f[1], (float)f[2], 0.f);
            }
            __syncthreads();
            for (int q0 = kSumBlock * sub; q0 < cnt; q0 += NS * kSumBlock) {
                const int qe = min(cnt, q0 + kSumBlock), pad = q0 / kSumBlock;
                float ux = 0.f, uy = 0.f, uz = 0.f;
#pragma unroll 4
                for (int q = q0 + pad; q < qe + pad; ++q) {
                    const float4 h = tile.h[q], l = tile.l[q];
                    float dx = hx - h.x, dy = hy - h.y, dz = hz - h.z;
                    float rxy2 = fmaf(dx, dx, dy * dy);
                    float r2 = fmaf(dz, dz, rxy2);
                    if (r2 < near2) {
                        const float4 o = tile.o[q];
                        dx += ox - o.x;
                        dy += oy - o.y;
                        dz += oz - o.z;
                        rxy2 = fmaf(dx, dx, dy * dy);
                        r2 = fmaf(dz, dz, rxy2);
                    }
                    if (WALL)
                        pair_wall_r2<float>(dx, dy, dz, rxy2, r2, hz + h.z, h.w, -hz, l.x, l.y, l.z, k, ux, uy, uz);
                    else
                        pair_free_r2<float>(dx, dy, dz, r2, l.x, l.y, l.z, k, ux, uy, uz);
                }
                two_sum_acc(th[0], tl[0], ux);
                two_sum_acc(th[1], tl[1], uy);
                two_sum_acc(th[2], tl[2], uz);
            }
        }
        s0 = (double)th[0] + (double)tl[0];
        s1 = (double)th[1] + (double)tl[1];
        s2 = (double)th[2] + (double)tl[2];
    }
    red[sub][0][e] = s0; red[sub][1][e] = s1; red[sub][2][e] = s2;
    __syncthreads();
    if (threadIdx.x < 3 * G) {
        const int c = threadIdx.x / G, t = threadIdx.x % G;
        double a = red[0][c][t];
        for (int q = 1; q < NS; ++q) a += red[q][c][t];
        own[3 * t + c] = a;
    }
    if (cs > 1) cluster_sync_all(); else __syncthreads();
    if (rank == 0 && threadIdx.x < 3 * G && group * G + (int)threadIdx.x / 3 < nt) {
        double a = own[threadIdx.x];
        for (int q = 1; q < cs; ++q) a += cluster_load(own + threadIdx.x, q);
        u[3 * (size_t)group * G + threadIdx.x] = k.A1 * a;
    }
    if (cs > 1) cluster_sync_all();  // the other CTAs' sums stay until they are read
}

// The FP32 product with two targets per thread (t0 + 64 group + e and + 32) in
// the lanes of float2 registers, positions already split into hi and lo
// (splitting them is FP64 work, repeated for every group); otherwise as
// k_rpy_small<float>, with the same blocks of 16 sources and pair terms that
// round alike, so both give the same result to the last bits of its 48-bit
// sums.
template <bool WALL>
__global__ void __launch_bounds__(kSmallThreads, 5)
k_rpy_small2(const float4* __restrict__ hi, const float4* __restrict__ lo, const double* __restrict__ lam,
              double* __restrict__ u, int n, int t0, int nt, int parts, RpyK<float> k) {
    dep_wait();
    constexpr int NS = kSmallThreads / 32;
    __shared__ float4 sq[3][kSmallTile];  // (-hx, -hx, -hy, -hy), (2hz, 2hz, lz, lz), (lx, lx, ly, ly)
    __shared__ float4 so[kSmallTile];     // (-ox, -ox, -oy, -oy)
    __shared__ float2 soz[kSmallTile];    // (-oz, -oz)
    __shared__ double red[NS][3][64];
    __shared__ double own[3 * 64];
    const int rank = (int)cluster_rank(), cs = (int)cluster_size();
    const int group = blockIdx.x / cs / parts, part = blockIdx.x / cs % parts;
    const int lane = threadIdx.x & 31, sub = threadIdx.x >> 5;
    const int nb = (n + kSumBlock - 1) / kSumBlock;
    const int piece = part * cs + rank, pieces = parts * cs;
    const int j0 = kSumBlock * (int)((long long)nb * piece / pieces);
    const int j1 = min(n, kSumBlock * (int)((long long)nb * (piece + 1) / pieces));
    u += (size_t)part * 3 * nt;
    float4 h0 = make_float4(0.f, 0.f, 1.f, 0.f), h1 = h0, o0 = make_float4(0.f, 0.f, 0.f, 0.f), o1 = o0;
    const int i0 = 64 * group + lane, i1 = i0 + 32;
    if (i0 < nt) { h0 = hi[t0 + i0]; o0 = lo[t0 + i0]; }
    if (i1 < nt) { h1 = hi[t0 + i1]; o1 = lo[t0 + i1]; }
    const float2 HX = make_float2(h0.x, h1.x), HY = make_float2(h0.y, h1.y), HZ = make_float2(h0.z, h1.z);
    const float2 LX = make_float2(o0.x, o1.x), LY = make_float2(o0.y, o1.y), LZ = make_float2(o0.z, o1.z);
    const float2 NX3 = make_float2(-h0.z, -h1.z);
    const float n0 = 0.25f * fmaxf(fabsf(h0.x), fmaxf(fabsf(h0.y), fabsf(h0.z)));
    const float n1 = 0.25f * fmaxf(fabsf(h1.x), fmaxf(fabsf(h1.y), fabsf(h1.z)));
    const float near2x = n0 * n0, near2y = n1 * n1;
    float2 hx = bc2(0.f), hy = bc2(0.f), hz = bc2(0.f), cx = bc2(0.f), cy = bc2(0.f), cz = bc2(0.f);
    for (int jt = j0; jt < j1; jt += kSmallTile) {
        const int cnt = min(kSmallTile, j1 - jt);
        __syncthreads();
        if ((int)threadIdx.x < cnt) {
            const int j = jt + threadIdx.x;
            const float4 h = hi[j], o = lo[j];
            const float lx = (float)lam[3 * (size_t)j], ly = (float)lam[3 * (size_t)j + 1],
                        lz = (float)lam[3 * (size_t)j + 2];
            sq[0][threadIdx.x] = make_float4(-h.x, -h.x, -h.y, -h.y);
            sq[1][threadIdx.x] = make_float4(2.f * h.z, 2.f * h.z, lz, lz);
            sq[2][threadIdx.x] = make_float4(lx, lx, ly, ly);
            so[threadIdx.x] = make_float4(-o.x, -o.x, -o.y, -o.y);
            soz[threadIdx.x] = make_float2(-o.z, -o.z);
        }
        __syncthreads();
        for (int q0 = kSumBlock * sub; q0 < cnt; q0 += NS * kSumBlock) {
            const int qe = min(cnt, q0 + kSumBlock);
            float2 ux = bc2(0.f), uy = bc2(0.f), uz = bc2(0.f);
#pragma unroll 2
            for (int q = q0; q < qe; ++q) {
                const float4 v0 = sq[0][q], v1 = sq[1][q], v2 = sq[2][q];
                const float2 h2 = make_float2(v1.x, v1.y);
                float2 dx = add2(HX, make_float2(v0.x, v0.y));
                float2 dy = add2(HY, make_float2(v0.z, v0.w));
                float2 dz = fma2(h2, bc2(-0.5f), HZ);
                const float2 Rz = fma2(h2, bc2(0.5f), HZ);
                float2 rxy2 = fma2(dx, dx, mul2(dy, dy));
                float2 r2 = fma2(dz, dz, rxy2);
                const bool na = r2.x < near2x, nb2 = r2.y < near2y;
                if (na || nb2) {  // lo parts where they matter, lane by lane
                    const float4 o = so[q];
                    const float2 ex = add2(dx, add2(LX, make_float2(o.x, o.y)));
                    const float2 ey = add2(dy, add2(LY, make_float2(o.z, o.w)));
                    const float2 ez = add2(dz, add2(LZ, soz[q]));
                    dx = make_float2(na ? ex.x : dx.x, nb2 ? ex.y : dx.y);
                    dy = make_float2(na ? ey.x : dy.x, nb2 ? ey.y : dy.y);
                    dz = make_float2(na ? ez.x : dz.x, nb2 ? ez.y : dz.y);
                    rxy2 = fma2(dx, dx, mul2(dy, dy));
                    r2 = fma2(dz, dz, rxy2);
                }
                pair2<WALL>(dx, dy, dz, rxy2, r2, Rz, h2, NX3, make_float2(v2.x, v2.y), make_float2(v2.z, v2.w),
                               make_float2(v1.z, v1.w), k, ux, uy, uz);
            }
            two_sum_acc2(hx, cx, ux);
            two_sum_acc2(hy, cy, uy);
            two_sum_acc2(hz, cz, uz);
        }
    }
    red[sub][0][lane] = (double)hx.x + (double)cx.x; red[sub][0][32 + lane] = (double)hx.y + (double)cx.y;
    red[sub][1][lane] = (double)hy.x + (double)cy.x; red[sub][1][32 + lane] = (double)hy.y + (double)cy.y;
    red[sub][2][lane] = (double)hz.x + (double)cz.x; red[sub][2][32 + lane] = (double)hz.y + (double)cz.y;
    __syncthreads();
    for (int e = threadIdx.x; e < 3 * 64; e += kSmallThreads) {
        const int c = e / 64, t = e % 64;
        double a = red[0][c][t];
        for (int q = 1; q < NS; ++q) a += red[q][c][t];
        own[3 * t + c] = a;
    }
    if (cs > 1) cluster_sync_all(); else __syncthreads();
    if (rank == 0)
        for (int e = threadIdx.x; e < 3 * 64 && 64 * group + e / 3 < nt; e += kSmallThreads) {
            double a = own[e];
            for (int q = 1; q < cs; ++q) a += cluster_load(own + e, q);
            u[3 * (size_t)64 * group + e] = k.A1 * a;
        }
    if (cs > 1) cluster_sync_all();
}

// Targets per CTA or cluster, CTAs per cluster and parts of the sources with
// slots of their own (at most `slots`; the sum is another launch) for nt targets
// against n sources, by the time (us) that they should take.  While all CTAs are
// resident the busiest SM's work counts (FP32: over the share of the pipe that so
// few CTAs keep busy; one CTA fills the FP64 pipe), beyond that the mean and most
// of a CTA more.  Clusters are not dealt out evenly (949 rows of 7,594 blobs, 150
// CTAs in clusters of 5: two on many of the 152 SMs, twice the time), so where
// they are not few they count as a less busy pipe.  Small products come out as
// one launch of clusters, large ones as single CTAs, 20 to 50 an SM.  Measured,
// FP64 wall, 2,135 rows of 17,086 blobs: one launch, 3.5 to 7 CTAs an SM, 5.18
// ms; parts, 10.6 4.77, 21 4.71, 56 (32 parts of groups of 8) 4.59; mixed, 4,271
// rows: 3.5 CTAs 242 us, 7 225, 21 205.
struct SmallCost {
    int g_min, g_max, per_thread, resident;  // targets per CTA: G x per_thread; CTAs an SM holds
    bool fp64;
    double pair, start, stage;  // us: a pair per thread of a CTA, a CTA, the staging of 128 sources
};
struct SmallShape {
    int G = 32, cs = 1, parts = 1;
    double us = 1e300;
};
inline SmallShape small_shape(int n, int nt, long long slots, const SmallCost& c) {
    SmallShape best;
    for (int parts : {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48}) {
        if (parts > 1 && (parts > slots || n / parts < 2 * kSmallTile)) break;
        const double sum = parts > 1 ? 5.0 + 1.2e-5 * parts * (double)nt : 0.0;
        for (int G = c.g_max; G >= c.g_min; G /= 2)
            for (int cs = 1; cs <= 8; ++cs) {
                if (parts > 1 && n / (parts * cs) < 2 * kSmallTile) break;
                const long long ctas = (long long)((nt + G * c.per_thread - 1) / (G * c.per_thread)) * cs * parts;
                const double mean = (double)ctas / num_sms(), most = std::ceil(mean);
                double load, start = c.start;
                if (cs == 1) {
                    const double busy = c.fp64 || most > 3.0 ? 1.0 : most > 2.0 ? 0.9 : most > 1.0 ? 0.76 : 0.47;
                    load = most <= c.resident ? (most > 1.0 ? 1.04 : 1.0) * most / busy : mean + 0.7;
                } else {
                    const double busy = c.fp64 && mean <= 0.9 ? 0.8 : std::max(0.4, std::min(1.0, 0.15 + 0.25 * mean));
                    load = (mean > 1.0 ? most * (0.99 + 0.01 * cs) + 0.25 : 1.0) / busy;
                    start = 4.0 * c.pair;
                }
                const double share = (double)((n + parts * cs - 1) / (parts * cs));
                const double us =
                    load * (std::ceil(share * G / kSmallThreads) * c.pair + start + share / kSmallTile * c.stage) + sum;
                if (us < best.us) best = {G, cs, parts, us};
            }
    }
    return best;
}

// Launch of a cluster kernel, as a programmatic dependent of the one before.
template <class K, class... Args>
inline void launch_cluster(K kernel, int groups, int cs, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cs;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    lc.gridDim = dim3((unsigned)(groups * cs));
    lc.blockDim = dim3(kSmallThreads);
    lc.stream = st;
    lc.attrs = at;
    lc.numAttrs = 2;
    cudaLaunchKernelEx(&lc, kernel, args...);
    count_launch();
}

template <class T, bool WALL>
inline void launch_small_t(const double* r, const double* lam, double* u, int n, int t0, int nt, const SmallShape& s,
                           const RpyK<T>& k, cudaStream_t st) {
    const int cl = (nt + s.G - 1) / s.G * s.parts;
    if (s.G == 32) launch_cluster(k_rpy_small<T, WALL, 32>, cl, s.cs, st, r, lam, u, n, t0, nt, s.parts, k);
    else if (s.G == 16) launch_cluster(k_rpy_small<T, WALL, 16>, cl, s.cs, st, r, lam, u, n, t0, nt, s.parts, k);
    else if constexpr (sizeof(T) == 8)
        launch_cluster(k_rpy_small<T, WALL, 8>, cl, s.cs, st, r, lam, u, n, t0, nt, s.parts, k);
}

}  // namespace am
