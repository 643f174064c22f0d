// Single-blob bodies with rotational coupling, free space (Sec. 2.4): every
// body is one blob of radius a at its tracking point, the body mobility N is
// the generalised RPY tensor (translation, rotation, and their coupling), and
// the constrained problem is Eq. linear_system_general on y = (U, phi):
//     U - N C^T phi = N F,     C U = B.
// Pair tensor for d = x_i - x_j, r = |d|, e = d / r (equal radii):
//   u_i     += M_tt(d) f_j + c(r) (T_j x e) ... written as -c(r) e x T_j
//   omega_i += -c(r) e x f_j + alpha(r) T_j + beta(r) (e . T_j) e
//   c     = 1 / (8 pi eta r^2)                         r >= 2a
//         = (r / a - 3 r^2 / (8 a^2)) / (16 pi eta a^2) r <  2a
//   alpha = -1 / (16 pi eta r^3),  beta = 3 / (16 pi eta r^3)          r >= 2a
//   alpha = (1 - 27 s / 32 + 5 s^3 / 64) / (8 pi eta a^3),
//   beta  = (9 s / 32 - 3 s^3 / 64) / (8 pi eta a^3),  s = r / a      r <  2a
//   self: mu0 = 1 / (6 pi eta a) for translation, 1 / (8 pi eta a^3) for
//   rotation (the far forms are the vorticity of the regularised Stokeslet
//   and of the rotlet; the overlapping ones are the closed forms for equal
//   spheres of Wajnryb, Mizerski, Zuk and Szymczak 2013).
// Preconditioner: N replaced by its self blocks N~ = diag(mu0 I, mu_r I), so
// phi = G~ (r_phi - C r_U) with G~ = (C N~ C^T)^+ per articulated body (the
// assembly factorisation of precond.cu) and U = r_U + N~ C^T phi.
#include "am_internal.cuh"
#include "ops.cuh"
#include "rpy_pair.cuh"
#include "sym_tiles.cuh"

#include <algorithm>

namespace am {

namespace {

// N~ of every body: diag(mu0 I3, mu_r I3) as 6 x 6 row-major
__global__ void k_sb_fill_nt(int M, double mu0, double mur, double* __restrict__ Nt) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= M) return;
    double* o = Nt + 36 * (size_t)p;
    for (int k = 0; k < 36; ++k) o[k] = 0.0;
    for (int k = 0; k < 3; ++k) { o[7 * k] = mu0; o[7 * (k + 3)] = mur; }
}

// (C^T phi)_p: +phi_n and l_p x phi_n on the link's body p, -phi_n and
// -(l_q x phi_n) on its body q (App. A)
__device__ __forceinline__ void ct_phi_body(int p, const int* __restrict__ blo, const int* __restrict__ bli,
                                            const double* __restrict__ lp, const double* __restrict__ lq,
                                            const double* __restrict__ phi, double* g) {
    for (int k = 0; k < 6; ++k) g[k] = 0.0;
    for (int e = blo[p]; e < blo[p + 1]; ++e) {
        const int code = bli[e], n = code >> 1, side = code & 1;
        const double f0 = phi[3 * (size_t)n], f1 = phi[3 * (size_t)n + 1], f2 = phi[3 * (size_t)n + 2];
        const double* l = side ? lq + 3 * (size_t)n : lp + 3 * (size_t)n;
        const double sg = side ? -1.0 : 1.0;
        g[0] += sg * f0; g[1] += sg * f1; g[2] += sg * f2;
        g[3] += sg * (l[1] * f2 - l[2] * f1);
        g[4] += sg * (l[2] * f0 - l[0] * f2);
        g[5] += sg * (l[0] * f1 - l[1] * f0);
    }
}

__global__ void k_sb_ctphi(int M, const int* __restrict__ blo, const int* __restrict__ bli,
                           const double* __restrict__ lp, const double* __restrict__ lq,
                           const double* __restrict__ phi, double* __restrict__ g) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= M) return;
    double v[6];
    ct_phi_body(p, blo, bli, lp, lq, phi, v);
    for (int k = 0; k < 6; ++k) g[6 * (size_t)p + k] = v[k];
}

// Both directions of one pair of bodies, velocities in units of A1 =
// 1/(8 pi eta), d = x_i - x_j unnormalised.  With ri = 1/r:
//   c1, c2 of the RPY tensor (rpy_pair.cuh);
//   the coupling c / (r A1) = ri^3                       r >= 2a
//                           = (1 - 3 s / 8) / (2 a^3)    r <  2a, s = r / a
//   alpha / A1 = -ri^3 / 2,  beta / (r^2 A1) = 3 ri^5 / 2     r >= 2a
//   alpha / A1 = (1 - 27 s / 32 + 5 s^3 / 64) / a^3,
//   beta / (r^2 A1) = (9 / (32 s) - 3 s / 64) / a^5           r <  2a
// (1/s taken as 0 at r = 0, where every term but the self mobilities
// vanishes).  FP64-issue-bound: about 90 FP64 operations per unordered pair
// (136 per ordered pair in the one-direction form with its divisions).
struct SymSpherePair : SymFp64 {
    static constexpr int kMinBlocks = 20;
    static constexpr int NC = 6;  // (force, torque) in, (velocity, rotation) out
    RpyK<double> k;
    double ia, h_a3, i_a3, n9_a4, n3_a5;  // 1/a, 1/(2 a^3), 1/a^3, 9/(32 a^4), -3/(64 a^5)
    __device__ __forceinline__ double scale() const { return k.A1; }
    __device__ __forceinline__ void both(const double* xi, const double* xj, const double* l, const double* m,
                                         double* u, double* v) const {
        const double dx = xi[0] - xj[0], dy = xi[1] - xj[1], dz = xi[2] - xj[2];
        const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
        double c1, c2, gc, al, be;
        if (r2 >= k.four_a2) {
            const double ri = rsq(r2);
            const double ri2 = ri * ri, ri3 = ri * ri2;
            c1 = ri * fma(k.kf2, ri2, 1.0);
            c2 = ri3 * fma(-k.kf3, ri2, 1.0);
            gc = ri3;
            al = -0.5 * ri3;
            be = 1.5 * (ri3 * ri2);
        } else {
            const double ri = r2 > 0.0 ? rsq(r2) : 0.0;
            const double sv = (r2 * ri) * ia, s2 = sv * sv;
            c1 = k.kn0 * fma(-k.kn1, r2 * ri, 1.0);
            c2 = k.kn2 * ri;
            gc = h_a3 * fma(-0.375, sv, 1.0);
            al = i_a3 * fma(fma(5.0 / 64.0, s2, -27.0 / 32.0), sv, 1.0);
            be = fma(n9_a4, ri, n3_a5 * sv);
        }
        const double gx = gc * dx, gy = gc * dy, gz = gc * dz;
        {
            const double sf = c2 * fma(dx, l[0], fma(dy, l[1], dz * l[2]));
            u[0] = fma(c1, l[0], fma(sf, dx, fma(gz, l[4], fma(-gy, l[5], u[0]))));
            u[1] = fma(c1, l[1], fma(sf, dy, fma(gx, l[5], fma(-gz, l[3], u[1]))));
            u[2] = fma(c1, l[2], fma(sf, dz, fma(gy, l[3], fma(-gx, l[4], u[2]))));
            const double st = be * fma(dx, l[3], fma(dy, l[4], dz * l[5]));
            u[3] = fma(al, l[3], fma(st, dx, fma(gz, l[1], fma(-gy, l[2], u[3]))));
            u[4] = fma(al, l[4], fma(st, dy, fma(gx, l[2], fma(-gz, l[0], u[4]))));
            u[5] = fma(al, l[5], fma(st, dz, fma(gy, l[0], fma(-gx, l[1], u[5]))));
        }
        {   // d and with it the coupling change sign
            const double sf = c2 * fma(dx, m[0], fma(dy, m[1], dz * m[2]));
            v[0] = fma(c1, m[0], fma(sf, dx, fma(-gz, m[4], fma(gy, m[5], v[0]))));
            v[1] = fma(c1, m[1], fma(sf, dy, fma(-gx, m[5], fma(gz, m[3], v[1]))));
            v[2] = fma(c1, m[2], fma(sf, dz, fma(-gy, m[3], fma(gx, m[4], v[2]))));
            const double st = be * fma(dx, m[3], fma(dy, m[4], dz * m[5]));
            v[3] = fma(al, m[3], fma(st, dx, fma(-gz, m[1], fma(gy, m[2], v[3]))));
            v[4] = fma(al, m[4], fma(st, dy, fma(-gx, m[2], fma(gz, m[0], v[4]))));
            v[5] = fma(al, m[5], fma(st, dz, fma(-gy, m[0], fma(gx, m[1], v[5]))));
        }
    }
    __device__ __forceinline__ void self(const double*, const double* m, double* u) const {
        for (int c = 0; c < 3; ++c) {
            u[c] = fma(k.kn0, m[c], u[c]);
            u[3 + c] = fma(i_a3, m[3 + c], u[3 + c]);
        }
    }
};

// v = the sum of the slots of the element's system (fixed order: 8 threads
// per element take every eighth slot)
__global__ void __launch_bounds__(256)
k_sb_sum(int n6, const int* __restrict__ sys_of_U, const int* __restrict__ sys_body_off,
         const long long* __restrict__ poff, const int* __restrict__ nslots, const double* __restrict__ part,
         double* __restrict__ v) {
    __shared__ double sh[8][32];
    const int e = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int t = blockIdx.x * 32 + e;
    double a = 0.0;
    if (t < n6) {
        const int s = sys_of_U[t], b0 = sys_body_off[s];
        const size_t n = 6 * (size_t)(sys_body_off[s + 1] - b0);
        const double* p = part + poff[s] + (t - 6 * (size_t)b0);
        const int ns = nslots[s];
#pragma unroll 4
        for (int c = q; c < ns; c += 8) a += p[c * n];
    }
    sh[q][e] = a;
    __syncthreads();
    if (q == 0 && t < n6) {
        for (int c = 1; c < 8; ++c) a += sh[c][e];
        v[t] = a;
    }
}

// out_U = U - v (v = N C^T phi); out_phi = C U
__global__ void k_sb_epilogue(int M, int P, const double* __restrict__ y, const double* __restrict__ v,
                              const int* __restrict__ bp, const int* __restrict__ bq,
                              const double* __restrict__ lp, const double* __restrict__ lq,
                              double* __restrict__ out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 6 * M) {
        out[t] = y[t] - v[t];
        return;
    }
    const int n = t - 6 * M;
    if (n >= P) return;
    const double* Up = y + 6 * (size_t)bp[n];
    const double* Uq = y + 6 * (size_t)bq[n];
    const double* l1 = lp + 3 * (size_t)n;
    const double* l2 = lq + 3 * (size_t)n;
    // u_p - l_p x omega_p - u_q + l_q x omega_q
    double* o = out + 6 * (size_t)M + 3 * (size_t)n;
    o[0] = Up[0] - (l1[1] * Up[5] - l1[2] * Up[4]) - Uq[0] + (l2[1] * Uq[5] - l2[2] * Uq[4]);
    o[1] = Up[1] - (l1[2] * Up[3] - l1[0] * Up[5]) - Uq[1] + (l2[2] * Uq[3] - l2[0] * Uq[5]);
    o[2] = Up[2] - (l1[0] * Up[4] - l1[1] * Up[3]) - Uq[2] + (l2[0] * Uq[4] - l2[1] * Uq[3]);
}

// z_U = r_U + N~ C^T phi (phi already in z)
__global__ void k_sb_ap3(int M, const int* __restrict__ blo, const int* __restrict__ bli,
                         const double* __restrict__ lp, const double* __restrict__ lq, double mu0, double mur,
                         const double* __restrict__ r, double* __restrict__ z) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= M) return;
    double g[6];
    ct_phi_body(p, blo, bli, lp, lq, z + 6 * (size_t)M, g);
    for (int k2 = 0; k2 < 6; ++k2) {
        const double s = k2 < 3 ? mu0 : mur;
        z[6 * (size_t)p + k2] = r[6 * (size_t)p + k2] + s * g[k2];
    }
}

inline int nb(long long n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

static double sb_mu0(const am_handle* h) { return 1.0 / (6.0 * 3.14159265358979323846 * h->cfg.eta * h->cfg.blob_radius); }
static double sb_mur(const am_handle* h) {
    const double a = h->cfg.blob_radius;
    return 1.0 / (8.0 * 3.14159265358979323846 * h->cfg.eta * a * a * a);
}

int sb_layout(am_handle* h) {
    long long tiles2 = 0;
    for (const auto& r : h->sys) {
        const long long ng = (r.M + 32LL * sym_group_tiles(r.M) - 1) / (32LL * sym_group_tiles(r.M));
        tiles2 += ng * (ng + 1) / 2;
    }
    const int splits = sym_step_splits(tiles2);
    std::vector<SymItem> items;
    std::vector<long long> poff(h->S);
    std::vector<int> nslots(h->S);
    long long off = 0;
    for (int s = 0; s < h->S; ++s) {
        const int n = h->sys[s].M;
        poff[s] = off;
        nslots[s] = sym_append_items(items, s, h->sys_body0[s], n, 6, sym_group_tiles(n), splits, off);
        off += 6LL * n * nslots[s];
    }
    sb_layout_free(h);
    cudaStream_t st = h->stream;
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sym_tiles<SymSpherePair>, 32 * kSymWarps, 0) !=
            cudaSuccess || per <= 0)
        per = 4;
    h->n_sb_items = (int)items.size();
    h->sb_grid = std::min(per * num_sms(), (h->n_sb_items + kSymWarps - 1) / kSymWarps);
    if (cudaMalloc(&h->d_sb_items, items.size() * sizeof(SymItem)) != cudaSuccess ||
        cudaMalloc(reinterpret_cast<void**>(&h->d_sbpart), off * sizeof(double)) != cudaSuccess ||
        cudaMalloc(reinterpret_cast<void**>(&h->d_sb_poff), h->S * sizeof(long long)) != cudaSuccess ||
        cudaMalloc(reinterpret_cast<void**>(&h->d_sb_nslots), h->S * sizeof(int)) != cudaSuccess ||
        cudaMemcpyAsync(h->d_sb_items, items.data(), items.size() * sizeof(SymItem), cudaMemcpyHostToDevice, st) !=
            cudaSuccess ||
        cudaMemcpyAsync(h->d_sb_poff, poff.data(), h->S * sizeof(long long), cudaMemcpyHostToDevice, st) !=
            cudaSuccess ||
        cudaMemcpyAsync(h->d_sb_nslots, nslots.data(), h->S * sizeof(int), cudaMemcpyHostToDevice, st) != cudaSuccess)
        return 1;
    return cudaStreamSynchronize(st) != cudaSuccess;
}

void sb_layout_free(am_handle* h) {
    for (void* p : {h->d_sb_items, (void*)h->d_sbpart, (void*)h->d_sb_poff, (void*)h->d_sb_nslots})
        if (p) cudaFree(p);
    h->d_sb_items = nullptr;
    h->d_sbpart = nullptr;
    h->d_sb_poff = nullptr;
    h->d_sb_nslots = nullptr;
    h->n_sb_items = 0;
}

// v = N g for all systems (block diagonal): the symmetric tile product of
// sym_tiles.cuh.  6,000 bodies: 7.80 -> 3.02 ms a product (one thread per
// target over every ordered pair before; the FP64 pipe needs about 2.6 ms for
// 90 operations per unordered pair).
void sb_mobility(am_handle* h, const double* g, double* v) {
    const double a = h->cfg.blob_radius, a3 = a * a * a, a4 = a3 * a;
    SymSpherePair pr;
    pr.k = rpy_consts<double>(h->prm);
    pr.ia = 1.0 / a;
    pr.h_a3 = 0.5 / a3;
    pr.i_a3 = 1.0 / a3;
    pr.n9_a4 = 9.0 / (32.0 * a4);
    pr.n3_a5 = -3.0 / (64.0 * a4 * a);
    launch_dep(k_sym_tiles<SymSpherePair>, dim3(h->sb_grid), dim3(32 * kSymWarps), 0, h->stream,
               (const double*)h->d_q, g, h->d_sbpart, static_cast<const SymItem*>(h->d_sb_items), h->n_sb_items,
               h->d_item_counter, pr, (const int*)nullptr, SymSpan{});
    k_sb_sum<<<nb(6LL * h->M, 32), 256, 0, h->stream>>>(6 * h->M, h->d_sys_of_elem, h->d_sys_body_off, h->d_sb_poff,
                                                        h->d_sb_nslots, h->d_sbpart, v);
    count_launch(2);
    long long pairs = 0;
    for (const auto& r : h->sys) pairs += (long long)r.M * r.M;
    h->pairs += pairs;
}

void sb_rhs(am_handle* h) {
    // b_U = N F (b_phi = B is already in place)
    sb_mobility(h, h->d_F, h->d_b);
}

void sb_op_apply(am_handle* h, const double* y, double* out) {
    cudaStream_t s = h->stream;
    const int M = h->M, P = h->P;
    if (P) {
        k_sb_ctphi<<<nb(M, 128), 128, 0, s>>>(M, h->d_body_link_off, h->d_body_link_idx, h->d_lp, h->d_lq,
                                              y + 6 * (size_t)M, h->d_pc_Uhat);
        count_launch();
        sb_mobility(h, h->d_pc_Uhat, h->d_dx);
    } else {
        cudaMemsetAsync(h->d_dx, 0, 6 * (size_t)M * sizeof(double), s);
    }
    k_sb_epilogue<<<nb(6LL * M + P, 256), 256, 0, s>>>(M, P, y, h->d_dx, h->d_bp, h->d_bq, h->d_lp, h->d_lq, out);
    count_launch();
}

void sb_pc_build(am_handle* h) {
    k_sb_fill_nt<<<nb(h->M, 128), 128, 0, h->stream>>>(h->M, sb_mu0(h), sb_mur(h), h->d_Nt);
    count_launch();
}

void sb_pc_apply(am_handle* h, const double* r, double* z) {
    cudaStream_t s = h->stream;
    const int M = h->M;
    // U^ = r_U
    cudaMemcpyAsync(h->d_pc_Uhat, r, 6 * (size_t)M * sizeof(double), cudaMemcpyDeviceToDevice, s);
    if (h->P) {
        pc_apply_links(h, r, z);  // phi = G~ (r_phi - C U^) into z
        k_sb_ap3<<<nb(M, 128), 128, 0, s>>>(M, h->d_body_link_off, h->d_body_link_idx, h->d_lp, h->d_lq,
                                            sb_mu0(h), sb_mur(h), r, z);
        count_launch();
    } else {
        cudaMemcpyAsync(z, r, 6 * (size_t)M * sizeof(double), cudaMemcpyDeviceToDevice, s);
    }
}

}  // namespace am
