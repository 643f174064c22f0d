// Block-diagonal preconditioner (Sec. 3.1): the exact solution of the
// approximate problem Eq. precond, where M keeps only same-body blocks M^(pp).
//
// Build, per body p (one block): M^(pp) from the pair tensors, its explicit
// inverse by blocked Cholesky, blocked triangular inverse and X^T X on 32 x 32
// shared-memory tiles, Y_p = (M^(pp))^-1 K_p, S_p = K_p^T Y_p and
// N~_p = S_p^-1 (bodies of more than two tiles take clusters of CTAs where that
// is expected to be faster; of many bodies of one shape, away from a wall, one is
// built and the others are rotated from it).  Per articulated body a (one
// block or cluster): H_a = C_a N~_a C_a^T and its generalised inverse G~_a
// (Eq. block_diag_const_res) by symmetric pivoted Cholesky (32-column panels,
// then the blocked inverse of the rank-r factor):
// H(perm) = L L^T with L of rank r gives
// G~ = perm [(L11 L11^T)^-1 0; 0 0] perm^T, which solves H phi = c exactly for
// every c in range(H) = range(C_a).
//
// Apply, for r = (r1, r2, r3):
//   w = M~^-1 r1;  U^ = N~ (-r2 - K^T w), with K^T w = Y^T r1
//   phi = G~ (r3 - C U^)
//   U = U^ + N~ C^T phi;  lambda = w + Y U  (= M~^-1 (r1 + K U)).
// The dense products run over flattened (body, 32-row chunk) and
// (articulated body, 32-row chunk) work items so that every SM gets work.
//
// Matrices are stored in T = double (FP64 path) or float (mixed path, where
// the preconditioner only steers the inner iterations); vectors are FP64.
#include "am_internal.cuh"
#include "dev_util.cuh"
#include "ops.cuh"
#include "rpy_pair.cuh"

#include <algorithm>

namespace am {

constexpr int kRows = 32;  // rows per apply work item

// One body per team: body_list[blockIdx.x / team size]; a cluster team
// splits the pair tensors, the tiles of the blocked inverse and the rows of
// Y among its CTAs, and its first CTA forms N~_p.
template <class T, class Team>
__global__ void __launch_bounds__(kPcThreads)
k_pcb_build(const int* __restrict__ body_list, const int* __restrict__ blob_off,
            const double4_32a* __restrict__ r4, const double4_32a* __restrict__ d4,
            const long long* __restrict__ moff, T* __restrict__ minv, T* __restrict__ work,
            T* __restrict__ Y, double* __restrict__ Nt, RpyK<T> prm, int wall, int* flags) {
    __shared__ double sh[64];
    __shared__ PcTiles<T> tiles;
    __shared__ int s_bad;
    const Team team;
    const int tr = team.rank(), ts = team.size();
    const int b = body_list[blockIdx.x / ts];
    const int i0 = blob_off[b];
    const int nbl = blob_off[b + 1] - i0;
    const int m = 3 * nbl;
    if (threadIdx.x == 0) s_bad = 0;
    T* A = minv + moff[b];
    T* L = work + 2 * moff[b];
    T* X = L + (size_t)m * m;
    // the lower triangle of M^(pp) (blob pairs ti >= sj, the factorisation
    // reads no entry above the diagonal), pair tensors in the storage
    // precision from FP64 differences
    for (int idx = threadIdx.x + tr * blockDim.x; idx < nbl * nbl; idx += blockDim.x * ts) {
        const int ti = idx / nbl, sj = idx % nbl;
        if (sj > ti) continue;
        const double4_32a x = r4[i0 + ti], y = r4[i0 + sj];
        T Tt[9];
        pair_tensor<T>((T)(x.x - y.x), (T)(x.y - y.y), (T)(x.z - y.z), (T)x.z, (T)y.z, prm, wall, Tt);
        for (int a = 0; a < 3; ++a)
            for (int c = 0; c < 3; ++c) L[(size_t)(3 * ti + a) * m + 3 * sj + c] = Tt[3 * a + c];
    }
    team.sync();
    // (M^(pp))^-1 by blocked Cholesky, triangular inverse and X^T X
    blocked_spd_inverse(L, X, A, m, tiles, &s_bad, team);
    if (s_bad) {
        if (threadIdx.x == 0 && tr == 0) atomicOr(flags, kFlagSingular);
        return;
    }
    T* Yb = Y + 18 * (size_t)i0;
    for (int i = threadIdx.x + tr * blockDim.x; i < m; i += blockDim.x * ts) {
        double y[6] = {0, 0, 0, 0, 0, 0};
        for (int bb = 0; bb < nbl; ++bb) {
            const double v[3] = {(double)A[(size_t)(3 * bb) * m + i], (double)A[(size_t)(3 * bb + 1) * m + i],
                                 (double)A[(size_t)(3 * bb + 2) * m + i]};
            const double4_32a dd = d4[i0 + bb];
            const double d[3] = {dd.x, dd.y, dd.z};
            double c[3];
            cross3(d, v, c);
            for (int a = 0; a < 3; ++a) { y[a] += v[a]; y[3 + a] += c[a]; }
        }
        for (int a = 0; a < 6; ++a) Yb[6 * (size_t)i + a] = (T)y[a];
    }
    team.sync();
    if (tr != 0) return;
    if (threadIdx.x < 36) {
        const int c = threadIdx.x / 6, e = threadIdx.x % 6;
        double s = 0.0;
        for (int bb = 0; bb < nbl; ++bb) {
            if (c < 3) {
                s += (double)Yb[6 * (size_t)(3 * bb + c) + e];
            } else {
                const double v[3] = {(double)Yb[6 * (size_t)(3 * bb) + e], (double)Yb[6 * (size_t)(3 * bb + 1) + e],
                                     (double)Yb[6 * (size_t)(3 * bb + 2) + e]};
                const double4_32a dd = d4[i0 + bb];
                const double d[3] = {dd.x, dd.y, dd.z};
                double cr[3];
                cross3(d, v, cr);
                s += cr[c - 3];
            }
        }
        sh[threadIdx.x] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double S[36];
        for (int k = 0; k < 36; ++k) S[k] = sh[k];
        if (!spd6_inverse(S, Nt + 36 * (size_t)b)) atomicOr(flags, kFlagSingular);
    }
}

// Q X Q^T of the 3 x 3 block X, rows ld entries apart
template <class T>
__device__ __forceinline__ void rotate_block(const T* q, const T* X, T* out, size_t ld) {
    T t[9];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const T x0 = X[j], x1 = X[ld + j], x2 = X[2 * ld + j];
#pragma unroll
        for (int i = 0; i < 3; ++i) t[3 * i + j] = q[3 * i] * x0 + q[3 * i + 1] * x1 + q[3 * i + 2] * x2;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            out[i * ld + j] = t[3 * i] * q[3 * j] + t[3 * i + 1] * q[3 * j + 1] + t[3 * i + 2] * q[3 * j + 2];
}

// Blocks of bodies that are rotations of a built one (without a wall M^(pp)
// turns with the body): with Q the rotation between them every 3 x 3 block of
// (M^(pp))^-1, Y and N~ becomes Q X Q^T.  Item: (body, built body, first blob,
// blobs).  Bound by FP64 issue (54 multiply-adds per blob pair) and the write of
// the factors; a factorisation costs m / 2 multiply-adds per entry.  216 bodies
// of 600 rows and 3,456 of 30 in FP64: every body built 56.5 ms, two built and
// the others rotated 7.1 + 1.05 ms; 2,240 bodies of 36 rows in FP32: 586 us,
// 105 + 27.
template <class T>
__global__ void __launch_bounds__(256)
k_pcb_copy(const int4* __restrict__ items, const int* __restrict__ blob_off, const double* __restrict__ theta,
           const long long* __restrict__ moff, T* __restrict__ minv, T* __restrict__ Y, double* __restrict__ Nt) {
    __shared__ double Q[9];
    const int4 it = items[blockIdx.x];
    const int b = it.x, a = it.y;
    if (threadIdx.x < 3) {  // column c of R_b R_a^T
        const int c = threadIdx.x;
        const double *ta = theta + 4 * (size_t)a, *tb = theta + 4 * (size_t)b;
        double x, y, z, ox, oy, oz;
        quat_rotate_inv(ta[0], ta[1], ta[2], ta[3], c == 0, c == 1, c == 2, x, y, z);
        quat_rotate(tb[0], tb[1], tb[2], tb[3], x, y, z, ox, oy, oz);
        Q[c] = ox; Q[3 + c] = oy; Q[6 + c] = oz;
    }
    __syncthreads();
    T q[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) q[k] = (T)Q[k];
    const int n = blob_off[b + 1] - blob_off[b];
    const size_t m = 3 * (size_t)n;
    const T* A = minv + moff[a];
    T* B = minv + moff[b];
    for (int idx = threadIdx.x; idx < it.w * n; idx += blockDim.x) {
        const size_t at = 3 * (size_t)(it.z + idx / n) * m + 3 * (idx % n);
        rotate_block(q, A + at, B + at, m);
    }
    for (int idx = threadIdx.x; idx < 2 * it.w; idx += blockDim.x) {
        const size_t at = 18 * (size_t)(it.z + idx / 2) + 3 * (idx % 2);
        rotate_block(q, Y + 18 * (size_t)blob_off[a] + at, Y + 18 * (size_t)blob_off[b] + at, 6);
    }
    if (it.z == 0 && threadIdx.x < 4) {
        const size_t at = 18 * (size_t)(threadIdx.x / 2) + 3 * (threadIdx.x % 2);
        rotate_block(Q, Nt + 36 * (size_t)a + at, Nt + 36 * (size_t)b + at, 6);
    }
}

// W = E N~ for E = sigma [I, -l^x] (3 x 6 block of C on one body, App. A)
__device__ __forceinline__ void e_times_n(double sg, const double* l, const double* N, double* W) {
    for (int c = 0; c < 6; ++c) {
        const double v[3] = {N[3 * 6 + c], N[4 * 6 + c], N[5 * 6 + c]};
        double cr[3];
        cross3(l, v, cr);
        for (int a = 0; a < 3; ++a) W[a * 6 + c] = sg * (N[a * 6 + c] - cr[a]);
    }
}

// One articulated body per team: asm_list[blockIdx.x / team size].  In a
// cluster team the first CTA takes the column steps of each panel (pivot
// search included) and the team shares the trailing tiles, the blocked inverse
// and the scatter into G~; the first CTA publishes the rank (or -1 while the
// factorisation goes on) in rank_out[a] before each team barrier, so every CTA
// leaves the panel loop at the same panel.
// Bound by the chain of column steps.  Rows and columns stay where they are:
// pos[i] is the place of row i in the pivot order, perm its inverse; a column
// step reads one row of H (kept transposed, so that it is the pivot's column),
// the panel's columns lie in shared memory (lay & 2: kNB m entries) by row, and
// every warp finds the pivot for itself with integer comparisons (FP64 ones
// cost 16 cycles of the SM each).  lay & 1: pos and perm in shared memory.
// 186 rows (31 rods, two links each): 771 (FP32) and 1,114 (FP64) us with rows and columns
// exchanged in global memory, 457 and 723 us so.
template <class T, class Team>
__global__ void __launch_bounds__(kPcThreads)
k_pca_build(const int* __restrict__ asm_list, const int* __restrict__ asm_link_off,
            const int* __restrict__ asm_link_idx, const int* __restrict__ bp, const int* __restrict__ bq,
            const double* __restrict__ lp, const double* __restrict__ lq, const double* __restrict__ Nt,
            const long long* __restrict__ goff, T* __restrict__ G, T* __restrict__ gwork,
            int* __restrict__ perm_all, int* __restrict__ pos_all, const long long* __restrict__ poff,
            int* __restrict__ rank_out, double tol, int mmax, int lay) {
    extern __shared__ unsigned char dyn_smem[];
    double* dg = reinterpret_cast<double*>(dyn_smem);  // m values: the Schur-complement diagonal
    __shared__ PcTiles<T> tiles;
    __shared__ double s_sk, s_isk;
    const Team team;
    const int tr = team.rank(), ts = team.size();
    const int a = asm_list[blockIdx.x / ts];
    const int L0 = asm_link_off[a];
    const int Pa = asm_link_off[a + 1] - L0;
    const int m = 3 * Pa;
    if (m == 0) return;
    const int lane = threadIdx.x & 31;
    T* H = gwork + 2 * goff[a];
    T* X = H + (size_t)m * m;  // column k of the factor in row k
    T* Ga = G + goff[a];
    int* perm = perm_all + poff[a];
    int* sperm = lay & 1 ? reinterpret_cast<int*>(dg + mmax) : perm;
    int* pos = lay & 1 ? sperm + mmax : pos_all + poff[a];
    T* const panel = lay & 2 ? reinterpret_cast<T*>(pos + mmax) : nullptr;
    for (int idx = threadIdx.x + tr * blockDim.x; idx < Pa * Pa; idx += blockDim.x * ts) {
        const int r = idx / Pa, c = idx % Pa;
        const int ln = asm_link_idx[L0 + r], lk = asm_link_idx[L0 + c];
        double blk[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        for (int sn = 0; sn < 2; ++sn) {
            const int bn = sn ? bq[ln] : bp[ln];
            for (int sk = 0; sk < 2; ++sk) {
                const int bk = sk ? bq[lk] : bp[lk];
                if (bn != bk) continue;
                double W[18];
                e_times_n(sn ? -1.0 : 1.0, sn ? lq + 3 * ln : lp + 3 * ln, Nt + 36 * (size_t)bn, W);
                const double* l = sk ? lq + 3 * lk : lp + 3 * lk;
                const double sg = sk ? -1.0 : 1.0;
                // (W E_k^T)[x][y] = sg (W[x][y] + (W[x][3:6] x l)_y)
                for (int x = 0; x < 3; ++x) {
                    const double w3[3] = {W[x * 6 + 3], W[x * 6 + 4], W[x * 6 + 5]};
                    double cr[3];
                    cross3(w3, l, cr);
                    for (int yy = 0; yy < 3; ++yy) blk[x * 3 + yy] += sg * (W[x * 6 + yy] + cr[yy]);
                }
            }
        }
        for (int x = 0; x < 3; ++x)
            for (int yy = 0; yy < 3; ++yy) H[(size_t)(3 * c + yy) * m + 3 * r + x] = (T)blk[x * 3 + yy];
    }
    team.sync();
    // symmetric pivoted Cholesky (largest remaining diagonal first, ties to
    // the lower place), stopped at the first pivot <= tol * the first one;
    // blocked: within a panel of 32 columns each column is formed from the
    // panel's earlier columns (left-looking) with the Schur-complement
    // diagonal dg kept up to date for the pivot search, and after the panel
    // the trailing block takes one tile-product update.
    if (tr == 0)
        for (int i = threadIdx.x; i < m; i += blockDim.x) {
            dg[i] = (double)H[(size_t)i * m + i];
            pos[i] = sperm[i] = i;
        }
    __syncthreads();
    unsigned long long thr = 0;  // bits of the threshold: positive doubles compare as integers
    int r = m;
    for (int k0 = 0; k0 < m; k0 += kNB) {
        const int kend = min(m, k0 + kNB);
        if (tr == 0) {
            T* Lp = panel ? panel : X + (size_t)k0 * m;
            bool stop = false;
            for (int k = k0; k < kend; ++k) {
                // pivot: every warp scans the remaining diagonal
                unsigned long long key = 0;
                unsigned at = 0xffffffffu;
                for (int i = lane; i < m; i += 32) {
                    const int q = pos[i];
                    unsigned long long v = (unsigned long long)__double_as_longlong(dg[i]);
                    if (v > 0x7ff0000000000000ull) v = 0;  // negative or NaN
                    if (q >= k && (v > key || (v == key && (unsigned)q < at))) { key = v; at = q; }
                }
                const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32));
                unsigned lo = (unsigned)(key >> 32) == hi ? (unsigned)key : 0u;
                lo = __reduce_max_sync(0xffffffffu, lo);
                const bool mine = key == (((unsigned long long)hi << 32) | lo);
                key = ((unsigned long long)hi << 32) | lo;
                at = __reduce_min_sync(0xffffffffu, mine ? at : 0xffffffffu);
                if (k == 0) thr = (unsigned long long)__double_as_longlong(tol * __longlong_as_double((long long)key));
                if (!(key > thr) || key == 0) { r = k; stop = true; break; }
                const int j = (int)at, p = sperm[j];
                if (threadIdx.x == 0) {
                    s_sk = sqrt(__longlong_as_double((long long)key));
                    s_isk = 1.0 / s_sk;
                }
                // column k: Schur value from the panel's earlier columns (at
                // most 31, summed in T), scaled by the pivot's inverse square
                // root (formed once)
                const int nk = k - k0;
                const T* row = H + (size_t)p * m;
                for (int base = 0; base < m; base += blockDim.x) {
                    const int i = base + threadIdx.x;
                    const bool live = i < m && pos[i] >= k;
                    T h = 0, acc = 0;
                    if (live) {
                        h = row[i];
#pragma unroll 8
                        for (int t = 0; t < nk; ++t) acc = fma(Lp[(size_t)t * m + i], Lp[(size_t)t * m + p], acc);
                    }
                    if (base == 0) __syncthreads();  // the root; every warp has searched
                    if (live) {
                        T v;
                        if (i == p) {
                            v = (T)s_sk;
                        } else {
                            const double l = ((double)h - (double)acc) * s_isk;
                            v = (T)l;
                            dg[i] -= l * l;
                        }
                        Lp[(size_t)nk * m + i] = v;
                        if (panel) X[(size_t)k * m + i] = v;
                    }
                }
                __syncthreads();
                if (threadIdx.x == 0 && j != k) {  // places k and j exchanged
                    const int o = sperm[k];
                    sperm[k] = p;
                    sperm[j] = o;
                    pos[p] = k;
                    pos[o] = j;
                }
                __syncthreads();
            }
            if (sperm != perm)
                for (int i = threadIdx.x; i < m; i += blockDim.x) perm[i] = sperm[i];
            if (threadIdx.x == 0) rank_out[a] = stop ? r : -1;
        }
        team.sync();
        const int st = *reinterpret_cast<volatile const int*>(rank_out + a);
        if (st >= 0) { r = st; break; }
        // trailing update of the rows and columns of places >= kend by the
        // panel's columns
        constexpr int E = kNB * kNB / kPcThreads;
        int q = 0;
        for (int i0 = kend; i0 < m; i0 += kNB) {
            for (int j0 = kend; j0 < m; j0 += kNB, ++q) {
                if (q % ts != tr) continue;
                for (int idx = threadIdx.x; idx < kNB * kNB; idx += blockDim.x) {
                    const int t = idx / kNB, x = idx % kNB;
                    const T* col = X + (size_t)(k0 + t) * m;
                    tiles.a[x][t] = i0 + x < m ? col[perm[i0 + x]] : (T)0;
                    tiles.b[x][t] = j0 + x < m ? col[perm[j0 + x]] : (T)0;
                }
                __syncthreads();
                T acc[E];
#pragma unroll
                for (int e = 0; e < E; ++e) acc[e] = 0;
                tile_mac<T, true>(tiles.b, tiles.a, acc);
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int c = acc_row(e), rr = acc_col(e);
                    if (i0 + rr < m && j0 + c < m) H[(size_t)perm[j0 + c] * m + perm[i0 + rr]] -= acc[e];
                }
                __syncthreads();
            }
        }
        team.sync();
    }
    // the leading r x r factor in pivot order, over H
    for (int idx = threadIdx.x + tr * blockDim.x; idx < r * r; idx += blockDim.x * ts) {
        const int i = idx % r, j = idx / r;
        if (j <= i) H[(size_t)i * m + j] = X[(size_t)j * m + perm[i]];
    }
    team.sync();
    if (threadIdx.x == 0 && tr == 0) rank_out[a] = r;
    // (L11 L11^T)^-1 of the rank-r leading block, blocked (written over H)
    blocked_chol_inverse(H, X, H, r, m, tiles, team);
    for (int idx = threadIdx.x + tr * blockDim.x; idx < m * m; idx += blockDim.x * ts) Ga[idx] = (T)0;
    team.sync();
    for (int idx = threadIdx.x + tr * blockDim.x; idx < r * r; idx += blockDim.x * ts) {
        const int i = idx / r, jj = idx % r;
        Ga[(size_t)perm[i] * m + perm[jj]] = H[(size_t)i * m + jj];
    }
}

// ------------------------------------------------------------- apply ---
// Work item it: body pcw_body[it], rows pcw_chunk[it]*32 .. +32.  128 threads:
// lane = row within the chunk, warp = quarter of the columns.  r1 is staged in
// shared memory in the storage precision: converting it at every use is FP64
// work (16 cycles of the SM per warp instruction) and was half of the time in
// FP32 (36,000 blobs, bodies of up to 600 rows: 105 us, now 45; the 144 MB of
// factors take 22 at the copy rate).
template <class T>
__global__ void __launch_bounds__(128)
k_pc_ap1(const int* __restrict__ pcw_body, const int* __restrict__ pcw_chunk,
         const int* __restrict__ blob_off, const T* __restrict__ minv,
         const long long* __restrict__ moff, const T* __restrict__ Y, const double* __restrict__ r,
         double* __restrict__ w, double* __restrict__ ytp, int Nb, const int* __restrict__ pcw_off,
         const double* __restrict__ Nt, double* __restrict__ Uhat, int* __restrict__ body_cnt) {
    dep_wait();
    constexpr int kStage = 1024;  // entries of r1 staged at a time
    __shared__ T rs[kStage];
    __shared__ double red[4][kRows];
    const int it = blockIdx.x;
    const int b = pcw_body[it];
    const int i0 = blob_off[b];
    const int m = 3 * (blob_off[b + 1] - i0);
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int row = pcw_chunk[it] * kRows + lane;
    const double* r1 = r + 3 * (size_t)i0;
    // eight independent loads in flight per thread, four partial sums
    T acc[4] = {0, 0, 0, 0};
    for (int c0 = 0; c0 < m; c0 += kStage) {
        const int cn = min(kStage, m - c0);
        __syncthreads();
        for (int k = threadIdx.x; k < cn; k += blockDim.x) rs[k] = (T)r1[c0 + k];
        __syncthreads();
        if (row < m) {
            const T* A = minv + moff[b] + (size_t)c0 * m + row;
            int k = part;
            for (; k + 28 < cn; k += 32) {
                T av[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) av[u] = A[(size_t)(k + 4 * u) * m];
#pragma unroll
                for (int u = 0; u < 8; ++u) acc[u & 3] = fma(av[u], rs[k + 4 * u], acc[u & 3]);
            }
            for (; k < cn; k += 4) acc[0] = fma(A[(size_t)k * m], rs[k], acc[0]);
        }
    }
    red[part][lane] = (double)((acc[0] + acc[1]) + (acc[2] + acc[3]));
    if (part == 3) {  // partial Y^T r1 over this chunk's rows
        double yv[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (row < m) {
            const T* Yr = Y + 18 * (size_t)i0 + 6 * (size_t)row;
            const double ri = r1[row];
#pragma unroll
            for (int c = 0; c < 6; ++c) yv[c] = (double)Yr[c] * ri;
        }
        const double t = warp_sums<8>(yv, lane);  // of column c in lanes 4 c .. 4 c + 3
        if (lane % 4 == 0 && lane < 24) ytp[6 * (size_t)it + lane / 4] = t;
    }
    __syncthreads();
    if (part == 0 && row < m) w[3 * (size_t)i0 + row] = red[0][lane] + red[1][lane] + red[2][lane] + red[3][lane];
    // the body's last item: U^_b = N~_b (-r2_b - sum of the body's Y^T r1
    // partials): lane 6 g + c adds every fifth partial of column c
    if (arrive_last(body_cnt, b, pcw_off[b + 1] - pcw_off[b]) && part == 0) {
        const int c = lane % 6, g = lane / 6;
        double v = 0.0;
        if (g < 5)
            for (int q = pcw_off[b] + g; q < pcw_off[b + 1]; q += 5) v += __ldcg(ytp + 6 * (size_t)q + c);
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < 5; ++q) s += __shfl_sync(0xffffffffu, v, 6 * q + c);
        v = lane < 6 ? -r[3 * (size_t)Nb + 6 * (size_t)b + lane] - s : 0.0;
        double vv[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) vv[q] = __shfl_sync(0xffffffffu, v, q);
        if (lane < 6) {
            const double* N = Nt + 36 * (size_t)b + 6 * lane;
            double t = 0.0;
#pragma unroll
            for (int q = 0; q < 6; ++q) t += N[q] * vv[q];
            Uhat[6 * (size_t)b + lane] = t;
        }
    }
}

// c_n = r3_n - (C U^)_n
__global__ void k_pc_cvec(int Nb, int M, int P, const int* __restrict__ bp, const int* __restrict__ bq,
                          const double* __restrict__ lp, const double* __restrict__ lq,
                          const double* __restrict__ Uhat, const double* __restrict__ r,
                          double* __restrict__ cbuf) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= P) return;
    const double* r3 = r + 3 * (size_t)Nb + 6 * (size_t)M;
    const double* up = Uhat + 6 * bp[n];
    const double* uq = Uhat + 6 * bq[n];
    double wp[3], wq[3];
    cross3(up + 3, lp + 3 * n, wp);
    cross3(uq + 3, lq + 3 * n, wq);
    for (int x = 0; x < 3; ++x) cbuf[3 * n + x] = r3[3 * n + x] - (up[x] + wp[x] - uq[x] - wq[x]);
}

// phi rows of one (articulated body, 32-row chunk) item: phi = G~ c, with c
// read from cbuf (k_pc_cvec) or, FUSED, formed here from U^ and r3 for the
// entries this block stages (c_n = r3_n - (C U^)_n)
template <class T, bool FUSED>
__global__ void __launch_bounds__(128)
k_pc_ap2(int Nb, int M, const int* __restrict__ pca_asm, const int* __restrict__ pca_chunk,
         const int* __restrict__ asm_link_off, const int* __restrict__ asm_link_idx,
         const T* __restrict__ G, const long long* __restrict__ goff, const double* __restrict__ cbuf,
         double* __restrict__ z, const int* __restrict__ bp, const int* __restrict__ bq,
         const double* __restrict__ lp, const double* __restrict__ lq, const double* __restrict__ Uhat,
         const double* __restrict__ r) {
    dep_wait();
    constexpr int kStage = 1024;  // entries of c staged in shared memory at a time
    __shared__ double red[4][kRows];
    __shared__ T cs[kStage];
    const int it = blockIdx.x;
    const int a = pca_asm[it];
    const int L0 = asm_link_off[a];
    const int m = 3 * (asm_link_off[a + 1] - L0);
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int row = pca_chunk[it] * kRows + lane;
    const T* Ga = G + goff[a];
    T acc[4] = {0, 0, 0, 0};
    for (int c0 = 0; c0 < m; c0 += kStage) {
        const int cn = min(kStage, m - c0);
        __syncthreads();
        for (int k = threadIdx.x; k < cn; k += blockDim.x) {
            const int kk = c0 + k;
            const int n = asm_link_idx[L0 + kk / 3], x = kk % 3;
            if (FUSED) {
                const double* up = Uhat + 6 * bp[n];
                const double* uq = Uhat + 6 * bq[n];
                double wp[3], wq[3];
                cross3(up + 3, lp + 3 * n, wp);
                cross3(uq + 3, lq + 3 * n, wq);
                cs[k] = (T)(r[3 * (size_t)Nb + 6 * (size_t)M + 3 * n + x] - (up[x] + wp[x] - uq[x] - wq[x]));
            } else {
                cs[k] = (T)cbuf[3 * n + x];
            }
        }
        __syncthreads();
        if (row < m) {
            const T* Gc = Ga + (size_t)c0 * m + row;
            int k = part;
            for (; k + 28 < cn; k += 32) {
                T gv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) gv[u] = Gc[(size_t)(k + 4 * u) * m];
#pragma unroll
                for (int u = 0; u < 8; ++u) acc[u & 3] = fma(gv[u], cs[k + 4 * u], acc[u & 3]);
            }
            for (; k < cn; k += 4) acc[0] = fma(Gc[(size_t)k * m], cs[k], acc[0]);
        }
    }
    const double s = row < m ? (double)((acc[0] + acc[1]) + (acc[2] + acc[3])) : 0.0;
    red[part][lane] = s;
    __syncthreads();
    if (part == 0 && row < m) {
        const int n = asm_link_idx[L0 + row / 3];
        z[3 * (size_t)Nb + 6 * (size_t)M + 3 * n + row % 3] = red[0][lane] + red[1][lane] + red[2][lane] + red[3][lane];
    }
}

// U_b = U^_b + N~_b (C^T phi)_b;  lambda rows = w + Y U, also as floats to lf
// when given.  A block per 128 rows (every fourth chunk): each block forms U_b
// for itself, which is more FP64 work than its rows.
template <class T>
__global__ void __launch_bounds__(128)
k_pc_ap3(int Nb, int M, const int* __restrict__ pcw_body, const int* __restrict__ pcw_chunk,
         const int* __restrict__ blob_off, const T* __restrict__ Y, const double* __restrict__ Nt,
         const double* __restrict__ w, const double* __restrict__ Uhat,
         const int* __restrict__ bl_off, const int* __restrict__ bl_idx,
         const double* __restrict__ lp, const double* __restrict__ lq, double* __restrict__ z,
         float* __restrict__ lf) {
    dep_wait();
    __shared__ double sU[6];
    const int it = blockIdx.x;
    if (pcw_chunk[it] % 4) return;
    const int b = pcw_body[it];
    const double* phi = z + 3 * (size_t)Nb + 6 * (size_t)M;
    if (threadIdx.x < 32) {
        // (C^T phi)_b: the body's link ends spread over the lanes of warp 0
        const int lane = threadIdx.x;
        double f[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int k = bl_off[b] + lane; k < bl_off[b + 1]; k += 32) {
            const int e = bl_idx[k];
            const int n = e >> 1;
            const double sg = (e & 1) ? -1.0 : 1.0;
            const double* l = (e & 1) ? lq + 3 * n : lp + 3 * n;
            const double* ph = phi + 3 * n;
            double t[3];
            cross3(l, ph, t);
            for (int x = 0; x < 3; ++x) { f[x] += sg * ph[x]; f[3 + x] += sg * t[x]; }
        }
        const double fs = warp_sums<8>(f, lane);  // of component c in lanes 4 c .. 4 c + 3
        double fc[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) fc[c] = __shfl_sync(0xffffffffu, fs, 4 * c);
        if (lane < 6) {
            const double* N = Nt + 36 * (size_t)b + 6 * lane;
            double s = Uhat[6 * (size_t)b + lane];
#pragma unroll
            for (int c = 0; c < 6; ++c) s += N[c] * fc[c];
            sU[lane] = s;
            if (pcw_chunk[it] == 0) z[3 * (size_t)Nb + 6 * (size_t)b + lane] = s;
        }
    }
    __syncthreads();
    const int i0 = blob_off[b];
    const int m = 3 * (blob_off[b + 1] - i0);
    const int row = pcw_chunk[it] * kRows + threadIdx.x;
    if (row < m) {
        const T* Yr = Y + 18 * (size_t)i0 + 6 * (size_t)row;
        double s = w[3 * (size_t)i0 + row];
        for (int c = 0; c < 6; ++c) s = fma((double)Yr[c], sU[c], s);
        z[3 * (size_t)i0 + row] = s;
        if (lf) lf[4 * (size_t)(i0 + row / 3) + row % 3] = (float)s;
    }
}

// The whole apply for handles of small articulated bodies (pc_small_size): one
// cluster per articulated body, a warp per body, one launch instead of three
// (the problem is block-diagonal over articulated bodies).  With n the body's
// rows (at most 36), lane l of the warp takes rows l and, when n > 32, the
// remaining rows with several lanes sharing each: an FP64 warp instruction
// costs 16 cycles of its SM however few lanes take part.  Every CTA forms c and
// phi of its articulated body itself (at most 64 rows of G~), so the cluster
// meets once.  Bound by chains of FP64 and L2 latency.  Measured, three kernels
// against this one: 4 chains of 8 bodies of 12 blobs in FP64 18.3 us against
// 14.0 (15.8 with a chain's bodies on the warps of one SM); 16 systems of 500 to
// 4,000 blobs in FP32 57 us against 22.
constexpr int kSmallRows = 64, kSmallBodyRows = 36;
template <class T>
__global__ void __launch_bounds__(256)
k_pc_small(int Nb, int M, const int* __restrict__ asm_body_off, const int* __restrict__ asm_body_idx,
           const int* __restrict__ asm_link_off, const int* __restrict__ asm_link_idx,
           const int* __restrict__ blob_off, const T* __restrict__ minv, const long long* __restrict__ moff,
           const T* __restrict__ Y, const double* __restrict__ Nt, const T* __restrict__ G,
           const long long* __restrict__ goff, const int* __restrict__ bp, const int* __restrict__ bq,
           const double* __restrict__ lp, const double* __restrict__ lq, const int* __restrict__ bl_off,
           const int* __restrict__ bl_idx, const int* __restrict__ link_local, const double* __restrict__ r,
           double* __restrict__ w, double* __restrict__ Uhat, double* __restrict__ z, float* __restrict__ lf) {
    dep_wait();
    __shared__ double phis[kSmallRows];
    __shared__ T ct[kSmallRows];
    __shared__ T red[8][kSmallRows];
    const ClusterTeam team;
    const int a = blockIdx.x / team.size();
    const int B0 = asm_body_off[a], Ma = asm_body_off[a + 1] - B0;
    const int L0 = asm_link_off ? asm_link_off[a] : 0, mg = asm_link_off ? 3 * (asm_link_off[a + 1] - L0) : 0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int wg = wid * team.size() + team.rank(), W = team.size() * 8;  // bodies spread over the SMs first
    // w = M~^-1 r1 and U^ = N~ (-r2 - Y^T r1)
    for (int q = wg; q < Ma; q += W) {
        const int b = asm_body_idx[B0 + q], i0 = blob_off[b], m = 3 * (blob_off[b + 1] - i0);
        const double* r1 = r + 3 * (size_t)i0;
        const T* A = minv + moff[b];
        const double ra = lane < m ? r1[lane] : 0.0, rb = 32 + lane < m ? r1[32 + lane] : 0.0;
        const T ta = (T)ra, tb = (T)rb;
        T acc0 = 0, acc1 = 0;
        for (int k = 0; k < m; k += 8) {  // rows 0 .. 31
            T av[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) av[u] = k + u < m && lane < m ? A[(size_t)(k + u) * m + lane] : (T)0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const T x = __shfl_sync(0xffffffffu, (k + u) & 32 ? tb : ta, (k + u) & 31);
                if (k + u < m) {
                    if (u & 1) acc1 = fma(av[u], x, acc1);
                    else acc0 = fma(av[u], x, acc0);
                }
            }
        }
        if (lane < m) w[3 * (size_t)i0 + lane] = (double)(acc0 + acc1);
        if (m > 32) {  // the remaining rows: `per` lanes on each column, 32 / per columns at a time
            const int rest = m - 32;
            int per = 1;
            while (per < rest) per *= 2;
            const int row = 32 + lane % per, k0 = lane / per, step = 32 / per;
            T t = 0;
#pragma unroll 4
            for (int k = 0; k < m; k += step) {
                const int kk = k + k0;
                const T xa = __shfl_sync(0xffffffffu, ta, kk & 31), xb = __shfl_sync(0xffffffffu, tb, kk & 31);
                if (kk < m && row < m) t = fma(A[(size_t)kk * m + row], kk & 32 ? xb : xa, t);
            }
            for (int o = per; o < 32; o *= 2) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane < rest) w[3 * (size_t)i0 + 32 + lane] = (double)t;
        }
        double yv[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (lane < m) {
            const T* Yr = Y + 18 * (size_t)i0 + 6 * lane;
#pragma unroll
            for (int c = 0; c < 6; ++c) yv[c] = (double)Yr[c] * ra;
        }
        if (32 + lane < m) {
            const T* Yr = Y + 18 * (size_t)i0 + 6 * (32 + lane);
#pragma unroll
            for (int c = 0; c < 6; ++c) yv[c] = fma((double)Yr[c], rb, yv[c]);
        }
        const double ys = warp_sums<8>(yv, lane);  // of column c in lanes 4 c .. 4 c + 3
        const double v = -(lane < 24 ? r[3 * (size_t)Nb + 6 * (size_t)b + lane / 4] : 0.0) - ys;
        // U^ = N~ v: lane 4 c + g takes columns g and g + 4 of row c
        const double* N = Nt + 36 * (size_t)b;
        const int c = lane >> 2, g = lane & 3;
        const double v0 = __shfl_sync(0xffffffffu, v, 4 * g), v1 = __shfl_sync(0xffffffffu, v, 4 * ((g + 4) % 6));
        double t = c < 6 ? N[6 * c + g] * v0 : 0.0;
        if (c < 6 && g < 2) t = fma(N[6 * c + g + 4], v1, t);
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        if (c < 6 && g == 0) Uhat[6 * (size_t)b + c] = t;
    }
    team.sync();
    // c = r3 - C U^ and phi = G~ c
    for (int k = threadIdx.x; k < mg; k += blockDim.x) {
        const int n = asm_link_idx[L0 + k / 3], x = k % 3, x1 = x == 2 ? 0 : x + 1, x2 = x == 0 ? 2 : x - 1;
        const double* up = Uhat + 6 * (size_t)bp[n];
        const double* uq = Uhat + 6 * (size_t)bq[n];
        const double *l1 = lp + 3 * (size_t)n, *l2 = lq + 3 * (size_t)n;
        // component x of u_p + omega_p x l_p - u_q - omega_q x l_q
        const double cp = __ldcg(up + x) + (__ldcg(up + 3 + x1) * l1[x2] - __ldcg(up + 3 + x2) * l1[x1]);
        const double cq = __ldcg(uq + x) + (__ldcg(uq + 3 + x1) * l2[x2] - __ldcg(uq + 3 + x2) * l2[x1]);
        ct[k] = (T)(r[3 * (size_t)Nb + 6 * (size_t)M + 3 * (size_t)n + x] - (cp - cq));
    }
    __syncthreads();
    if (mg) {
        const T* Ga = G + goff[a];
        for (int row = lane; row < mg; row += 32) {  // warp w: columns w, w + 8, ..
            T t = 0;
#pragma unroll 8
            for (int k = wid; k < mg; k += 8) t = fma(Ga[(size_t)k * mg + row], ct[k], t);
            red[wid][row] = t;
        }
        __syncthreads();
        if (threadIdx.x < mg) {
            double t = 0.0;
            for (int q = 0; q < 8; ++q) t += (double)red[q][threadIdx.x];
            phis[threadIdx.x] = t;
            if (team.rank() == 0) {
                const int n = asm_link_idx[L0 + threadIdx.x / 3];
                z[3 * (size_t)Nb + 6 * (size_t)M + 3 * (size_t)n + threadIdx.x % 3] = t;
            }
        }
        __syncthreads();
    }
    // U = U^ + N~ C^T phi; lambda = w + Y U
    for (int q = wg; q < Ma; q += W) {
        const int b = asm_body_idx[B0 + q], i0 = blob_off[b], m = 3 * (blob_off[b + 1] - i0);
        double f[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (mg)
            for (int k = bl_off[b] + lane; k < bl_off[b + 1]; k += 32) {
                const int e = bl_idx[k], n = e >> 1;
                const double sg = (e & 1) ? -1.0 : 1.0;
                const double* l = (e & 1) ? lq + 3 * (size_t)n : lp + 3 * (size_t)n;
                const double* ph = phis + 3 * link_local[n];
                const double p0 = sg * ph[0], p1 = sg * ph[1], p2 = sg * ph[2];
                f[0] += p0; f[1] += p1; f[2] += p2;
                f[3] = fma(l[1], p2, fma(-l[2], p1, f[3]));
                f[4] = fma(l[2], p0, fma(-l[0], p2, f[4]));
                f[5] = fma(l[0], p1, fma(-l[1], p0, f[5]));
            }
        const double fs = mg ? warp_sums<8>(f, lane) : 0.0;
        const double* N = Nt + 36 * (size_t)b;
        const int c = lane >> 2, g = lane & 3;
        const double f0 = __shfl_sync(0xffffffffu, fs, 4 * g), f1 = __shfl_sync(0xffffffffu, fs, 4 * ((g + 4) % 6));
        double t = c < 6 ? N[6 * c + g] * f0 : 0.0;
        if (c < 6 && g < 2) t = fma(N[6 * c + g + 4], f1, t);
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        if (c < 6) t += __ldcg(Uhat + 6 * (size_t)b + c);
        if (c < 6 && g == 0) z[3 * (size_t)Nb + 6 * (size_t)b + c] = t;
        double u[6];
#pragma unroll
        for (int x = 0; x < 6; ++x) u[x] = __shfl_sync(0xffffffffu, t, 4 * x);
        for (int row = lane; row < m; row += 32) {
            const T* Yr = Y + 18 * (size_t)i0 + 6 * row;
            double v = __ldcg(w + 3 * (size_t)i0 + row);
#pragma unroll
            for (int x = 0; x < 6; ++x) v = fma((double)Yr[x], u[x], v);
            z[3 * (size_t)i0 + row] = v;
            if (lf) lf[4 * (size_t)(i0 + row / 3) + row % 3] = (float)v;
        }
    }
}

// ----------------------------------------------------------------- host ---
// Launch of a build kernel over the items list[0 .. n): one CTA each, or
// one cluster of cs CTAs each.
template <class K, class... Args>
static void launch_team(K kernel, int n, int cs, size_t smem, cudaStream_t s, Args... args) {
    if (n <= 0) return;
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    lc.gridDim = dim3((unsigned)(n * cs));
    lc.blockDim = dim3(kPcThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    lc.attrs = at;
    lc.numAttrs = cs > 1 ? 1 : 0;
    cudaLaunchKernelEx(&lc, kernel, args...);
    count_launch();
}

template <class T>
static void pca_build_t(am_handle* h, double tol) {
    // the Schur diagonal and, as far as they fit, the places and the panel.  64 KB
    // beside the tiles leave an SM the two CTAs that its registers allow (4,000
    // articulated bodies of 6 rows beside one of 9, 87, 177 or 417 rows: 615 us in
    // FP64, 420 in FP32, whatever the longest); a larger panel stays in global memory
    const int m = 3 * std::max(1, h->max_asm_links);
    size_t smem = (size_t)m * sizeof(double);
    int lay = 0;
    if (2 * smem <= 160 * 1024) {
        lay = 1;
        smem *= 2;
        if (smem + (size_t)kNB * m * sizeof(T) <= 64 * 1024) {
            lay = 3;
            smem += (size_t)kNB * m * sizeof(T);
        }
    }
    if (smem > 16 * 1024) {
        cudaFuncSetAttribute(k_pca_build<T, CtaTeam>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(k_pca_build<T, ClusterTeam>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    }
    const int n_one = h->pca_cs > 1 ? h->n_pca_small : h->NA;
    launch_team(k_pca_build<T, CtaTeam>, n_one, 1, smem, h->stream, (const int*)h->d_pca_list,
                (const int*)h->d_asm_link_off, (const int*)h->d_asm_link_idx, (const int*)h->d_bp,
                (const int*)h->d_bq, (const double*)h->d_lp, (const double*)h->d_lq, (const double*)h->d_Nt,
                (const long long*)h->d_G_off, (T*)h->d_G, (T*)h->d_Gwork, h->d_perm,
                h->d_pos, (const long long*)h->d_perm_off, h->d_G_rank, tol, m, lay);
    if (h->pca_cs > 1)
        launch_team(k_pca_build<T, ClusterTeam>, h->NA - h->n_pca_small, h->pca_cs, smem, h->stream,
                    (const int*)(h->d_pca_list + h->n_pca_small), (const int*)h->d_asm_link_off,
                    (const int*)h->d_asm_link_idx, (const int*)h->d_bp, (const int*)h->d_bq,
                    (const double*)h->d_lp, (const double*)h->d_lq, (const double*)h->d_Nt,
                    (const long long*)h->d_G_off, (T*)h->d_G, (T*)h->d_Gwork, h->d_perm,
                    h->d_pos, (const long long*)h->d_perm_off, h->d_G_rank, tol, m, lay);
}

// Whether every articulated body is small enough for k_pc_small, and the
// cluster size: a warp per body, as many CTAs as spread them over the SMs.
// Measured against the three kernels, per GMRES iteration: bodies of 12 rows 2
// to 5 us less, of 36 rows 4 less to 1 more, of 42 rows 1 to 4 more, of 54 to 63
// rows 4 to 10 more (one warp walks a body's factors; the three kernels have a
// CTA per 32 rows).  Each articulated body has a CTA of eight warps: of one
// body each, 600 of them 3 us less, 800 3 more, 3,000 10 more; of two, 600 4 to 8
// less, 1,500 5 to 11 more; of four, 1,500 no more.  Periodic handles, whose
// iterations take milliseconds, keep the three kernels that they were measured with.
static int pc_small_size(const am_handle* h) {
    if (h->sb || h->per || h->NA == 0) return 0;
    if (3 * h->max_body_blobs > kSmallBodyRows || (h->P && 3 * h->max_asm_links > kSmallRows)) return 0;
    if (h->NA > 4 * num_sms() && h->M < 4 * h->NA) return 0;
    int most = 0;
    for (int a = 0; a < h->NA; ++a) most = std::max(most, h->asm_body_off[a + 1] - h->asm_body_off[a]);
    if (most > 64) return 0;
    int cs = 1;
    while (cs < 8 && cs < most && 2LL * cs * h->NA <= num_sms()) cs *= 2;
    return cs;
}

template <class T>
static void pc_build_t(am_handle* h, double tol) {
    cudaStream_t s = h->stream;
    // one block of kPcThreads per body and per articulated body (the tile
    // routines assume that block size)
    // bodies of one or two 32-row tiles one CTA each; larger bodies one
    // cluster of pcb_cs CTAs each
    const int n_one = h->pcb_cs > 1 ? h->n_pcb_small : h->n_pcb;
    launch_team(k_pcb_build<T, CtaTeam>, n_one, 1, 0, s, (const int*)h->d_pcb_list, (const int*)h->d_blob_off,
                (const double4_32a*)h->d_r4, (const double4_32a*)h->d_d4, (const long long*)h->d_minv_off,
                (T*)h->d_minv, (T*)h->d_pcwork, (T*)h->d_Y, h->d_Nt, rpy_consts<T>(h->prm), h->cfg.wall,
                h->d_flags);
    if (h->pcb_cs > 1)
        launch_team(k_pcb_build<T, ClusterTeam>, h->n_pcb - h->n_pcb_small, h->pcb_cs, 0, s,
                    (const int*)(h->d_pcb_list + h->n_pcb_small), (const int*)h->d_blob_off,
                    (const double4_32a*)h->d_r4, (const double4_32a*)h->d_d4, (const long long*)h->d_minv_off,
                    (T*)h->d_minv, (T*)h->d_pcwork, (T*)h->d_Y, h->d_Nt, rpy_consts<T>(h->prm),
                    h->cfg.wall, h->d_flags);
    if (h->n_pcb_copy) {
        k_pcb_copy<T><<<h->n_pcb_copy, 256, 0, s>>>(h->d_pcb_copy, h->d_blob_off, h->d_theta, h->d_minv_off,
                                                    (T*)h->d_minv, (T*)h->d_Y, h->d_Nt);
        count_launch();
    }
    if (h->P) pca_build_t<T>(h, tol);
}

void pc_apply_links(am_handle* h, const double* r, double* z) {
    cudaStream_t s = h->stream;
    k_pc_cvec<<<(h->P + 127) / 128, 128, 0, s>>>(h->Nb, h->M, h->P, h->d_bp, h->d_bq, h->d_lp, h->d_lq,
                                                  h->d_pc_Uhat, r, h->d_cbuf);
    if (h->pc32)
        k_pc_ap2<float, false><<<h->n_pca, 128, 0, s>>>(h->Nb, h->M, h->d_pca_asm, h->d_pca_chunk,
                                                         h->d_asm_link_off, h->d_asm_link_idx, (const float*)h->d_G,
                                                         h->d_G_off, h->d_cbuf, z, nullptr, nullptr, nullptr,
                                                         nullptr, nullptr, nullptr);
    else
        k_pc_ap2<double, false><<<h->n_pca, 128, 0, s>>>(h->Nb, h->M, h->d_pca_asm, h->d_pca_chunk,
                                                          h->d_asm_link_off, h->d_asm_link_idx, (const double*)h->d_G,
                                                          h->d_G_off, h->d_cbuf, z, nullptr, nullptr, nullptr,
                                                          nullptr, nullptr, nullptr);
    count_launch(2);
}

void pc_build(am_handle* h) {
    // arrival counts of the apply's per-body reductions (each completing
    // block zeroes its own; zeroed here as well, outside any graph)
    if (h->d_pcb_cnt) cudaMemsetAsync(h->d_pcb_cnt, 0, std::max(h->M, 1) * sizeof(int), h->stream);
    h->pc_small_cs = pc_small_size(h);
    if (h->sb) {
        sb_pc_build(h);
        if (h->P) pca_build_t<double>(h, 1e-11);
        h->pc_valid = true;
        return;
    }
    if (h->pc32)
        pc_build_t<float>(h, 1e-5);
    else
        pc_build_t<double>(h, 1e-11);
    h->pc_valid = true;
}

template <class T>
static void pc_apply_t(am_handle* h, const double* r, double* z, float* lf) {
    cudaStream_t s = h->stream;
    if (h->pc_small_cs) {
        cudaLaunchConfig_t lc = {};
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        at[1].id = cudaLaunchAttributeClusterDimension;
        at[1].val.clusterDim.x = (unsigned)h->pc_small_cs;
        at[1].val.clusterDim.y = 1;
        at[1].val.clusterDim.z = 1;
        lc.gridDim = dim3((unsigned)(h->NA * h->pc_small_cs));
        lc.blockDim = dim3(256);
        lc.stream = s;
        lc.attrs = at;
        lc.numAttrs = 2;
        cudaLaunchKernelEx(&lc, k_pc_small<T>, h->Nb, h->M, (const int*)h->d_asm_body_off,
                           (const int*)h->d_asm_body_idx, h->P ? (const int*)h->d_asm_link_off : (const int*)nullptr,
                           (const int*)h->d_asm_link_idx, (const int*)h->d_blob_off, (const T*)h->d_minv,
                           (const long long*)h->d_minv_off, (const T*)h->d_Y, (const double*)h->d_Nt,
                           (const T*)h->d_G, (const long long*)h->d_G_off, (const int*)h->d_bp, (const int*)h->d_bq,
                           (const double*)h->d_lp, (const double*)h->d_lq, (const int*)h->d_body_link_off,
                           (const int*)h->d_body_link_idx, (const int*)h->d_link_local, r, h->d_pc_w, h->d_pc_Uhat,
                           z, lf);
        count_launch();
        return;
    }
    // w and Y^T r1 per (body, chunk) item; the body's last item forms U^
    launch_dep(k_pc_ap1<T>, dim3(h->n_pcw), dim3(128), 0, s, h->d_pcw_body, h->d_pcw_chunk, h->d_blob_off,
               (const T*)h->d_minv, h->d_minv_off, (const T*)h->d_Y, r, h->d_pc_w, h->d_ytp, h->Nb, h->d_pcw_off,
               h->d_Nt, h->d_pc_Uhat, h->d_pcb_cnt);
    count_launch();
    if (h->P) {
        // phi = G~ (r3 - C U^), c formed per staged entry
        launch_dep(k_pc_ap2<T, true>, dim3(h->n_pca), dim3(128), 0, s, h->Nb, h->M, h->d_pca_asm, h->d_pca_chunk,
                   h->d_asm_link_off, h->d_asm_link_idx, (const T*)h->d_G, h->d_G_off, nullptr, z, h->d_bp, h->d_bq,
                   h->d_lp, h->d_lq, h->d_pc_Uhat, r);
        count_launch();
    }
    launch_dep(k_pc_ap3<T>, dim3(h->n_pcw), dim3(128), 0, s, h->Nb, h->M, h->d_pcw_body, h->d_pcw_chunk,
               h->d_blob_off, (const T*)h->d_Y, h->d_Nt, h->d_pc_w, h->d_pc_Uhat, h->d_body_link_off,
               h->d_body_link_idx, h->d_lp, h->d_lq, z, lf);
    count_launch();
}

void pc_apply(am_handle* h, const double* r, double* z, float4* lf) {
    if (h->sb) {
        sb_pc_apply(h, r, z);
        return;
    }
    if (h->pc32)
        pc_apply_t<float>(h, r, z, reinterpret_cast<float*>(lf));
    else
        pc_apply_t<double>(h, r, z, reinterpret_cast<float*>(lf));
}

}  // namespace am
