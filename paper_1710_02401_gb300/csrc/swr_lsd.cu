// swr_lsd.cu -- local orbitals (LOs) and local Slater determinants (LSDs).
//
// The paper's second basis family (Sec. 3.2 "Local orbital construction",
// Eq. BARPOT, Eq. LSD; Appendix A "Discrete local Hamiltonian construction
// with local Slater's determinants"; Sec. 7 Test 1 and its Table 1):
//
//   1. in every 1-D subdomain D_i the one-electron eigenproblem
//        1/2 int a phi' psi' + int (V_en + V_b) phi psi = lambda int phi psi,
//      V_b = V_inf s(|x - x_ci| - x_b), a = 1 - s, s the C^2 step rising over
//      [x_b - eps_b/2, x_b + eps_b/2], in a Gaussian basis of kd functions:
//      quadrature of the overlap and Hamiltonian matrices, Cholesky of the
//      overlap, parallel cyclic Jacobi of L^-1 H L^-T in shared memory, back
//      substitution, the M lowest orbitals, each with the sign that makes
//      int phi(x) exp(0.37 (x - x_ci)) dx positive (one CTA per subdomain);
//   2. every orbital at the nodes of one composite Gauss-Legendre rule over
//      the line, and the one-electron integrals between all orbitals:
//      <phi_a, phi_b>, 1/2 <phi_a', phi_b'> + <phi_a|V_en|phi_b>, <phi_a|x|phi_b>
//      (Appendix A's I and J);
//   3. the pair densities w phi_a phi_c of orbitals whose supports
//      [x_ci - x_b - m, x_ci + x_b + m] meet (m past the Gaussian tails; the
//      same or neighbouring subdomains for x_b near |D_i| / 2), T = P W with the soft-Coulomb
//      kernel W(x, s), so that the two-electron integral (ac|bd) of
//      Appendix A is the dot product of T_ac and P_bd;
//   4. per 2-D subdomain Omega_{i,j} (x1 in D_i, x2 in D_j) the K
//      determinants of lowest lambda_l^i + lambda_p^j (l < p when i = j; sums
//      within 1e-9 relative are ties broken by (l, p)), their Gram matrix
//      <a,c><b,d> - <a,d><b,c>, the matrix of H0 = h(1) + h(2) + W(x1 - x2):
//      h_ac S_bd + S_ac h_bd - h_ad S_bc - S_ad h_bc + (ac|bd) - (ad|bc), and
//      their Gram against the determinants of Omega_{i+1,j} (Table 1's w).
//
// Nuclear and electron-electron interactions are soft-Coulomb (the 1-D
// mollified Coulomb of Eq. GEPS diverges).  All arithmetic is FP64; every
// reduction has a fixed order.  The host only lays out the quadrature panels
// and the index tables.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "swr_internal.cuh"

namespace swr {

#define LSD_KD_MAX 64
#define LSD_Q_MAX 16
#define LSD_TIE 1e-9

struct LsdDev {
    double a, H, eps, xb, eps_b, v_inf, delta, eta_en, eta_ee, ee_coef, harmonic;
    double xn[3], zn[3];
    int L, M, K, kd, q, n_nuc, ng, n_pairs;
};

__device__ inline double lsd_centre(const LsdDev& d, int i) { return d.a + (i + 0.5) * d.H; }

// C^2 step: 0 for u <= 0, 1 for u >= 1, 6u^5 - 15u^4 + 10u^3 between.
__device__ inline double lsd_step(double u) {
    u = fmin(fmax(u, 0.0), 1.0);
    return u * u * u * (u * (6.0 * u - 15.0) + 10.0);
}
__device__ inline double lsd_switch(const LsdDev& d, double x, double xc) {
    const double t = fabs(x - xc) - d.xb;
    return lsd_step((t + 0.5 * d.eps_b) / d.eps_b);
}
__device__ inline double lsd_ven(const LsdDev& d, double x) {
    double v = 0.5 * d.harmonic * x * x;
    for (int A = 0; A < d.n_nuc; ++A) v -= d.zn[A] / sqrt((x - d.xn[A]) * (x - d.xn[A]) + d.eta_en * d.eta_en);
    return v;
}

// Gauss-Legendre nodes and weights of order q on [-1, 1]: Newton's method on
// the three-term recurrence of P_q, from the Chebyshev-like initial guess.
__global__ void k_lsd_gl(int q, double* t, double* w) {
    const int k = threadIdx.x;
    if (k >= q) return;
    double x = cos(3.14159265358979323846 * (k + 0.75) / (q + 0.5)), dp = 1.0, last = 1.0;
    for (int it = 0; it < 100; ++it) {
        double p0 = 1.0, p1 = x;
        for (int j = 2; j <= q; ++j) {
            const double p2 = ((2.0 * j - 1.0) * x * p1 - (j - 1.0) * p0) / j;
            p0 = p1;
            p1 = p2;
        }
        dp = q * (x * p1 - p0) / (x * x - 1.0);
        const double dx = p1 / dp;
        x -= dx;
        if (last < 1e-8) break;  // quadratic convergence: this step was the last that changes x
        last = fabs(dx);
    }
    t[q - 1 - k] = x;  // ascending
    w[q - 1 - k] = 2.0 / ((1.0 - x * x) * dp * dp);
}

// Nodes of composite rules: panel p of [edges[p], edges[p+1]] gives nodes
// p q .. p q + q - 1 (panels of all rules concatenated, edge index base[p]).
__global__ void k_lsd_nodes(const double* edges, const int* ebase, int n_panels, const double* t, const double* w, int q,
                            double* x, double* wx) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= n_panels * q) return;
    const int p = n / q, k = n - p * q;
    const double e0 = edges[ebase[p]], e1 = edges[ebase[p] + 1];
    x[n] = 0.5 * (e1 - e0) * t[k] + 0.5 * (e1 + e0);
    wx[n] = 0.5 * (e1 - e0) * w[k];
}

// ------------------------------------------------------ 1. local orbitals
//
// Three kernels: Gaussians and weights at the local nodes (one thread per
// value: every exponential, square root and barrier switch evaluated once),
// the overlap and Hamiltonian entries (one warp per entry of the upper
// triangle, lanes over the nodes), and the dense eigenproblem (one CTA per
// subdomain).  FP64 runs at 1.6 multiply-adds per clock on an SM of this
// part, so what one CTA does alone is kept to the O(kd^3) of the
// eigenproblem: with the quadrature inside that CTA (potential and switch per
// entry and node) the L = 5, M = 10, kd = 40 build took 25.5 ms in this
// stage, now 1.07 ms (1.03 of it the eigenproblem: ~350 Jacobi rounds bound by
// the FP64 pipe of one SM and two barriers each); whole call 27.3 -> 2.0 ms.

// Table rows of subdomain i, each nn nodes long: kd rows of g_k, kd rows of
// g_k', then w, 1/2 w a, w (V_en + V_b) and w exp(0.37 (x - x_ci)).
#define LSD_WROWS 4
__host__ __device__ inline size_t lsd_tab0(int n0, int kd) { return (size_t)n0 * (2 * kd + LSD_WROWS); }

__global__ void k_lsd_local_tab(LsdDev d, const double* xl, const double* wl, const int* nbase, double* gtab) {
    const int i = blockIdx.y, kd = d.kd, n0 = nbase[i], nn = nbase[i + 1] - n0;
    const double xc = lsd_centre(d, i), h = 2.0 * d.xb / (kd - 1);
    double* g = gtab + lsd_tab0(n0, kd);
    double* dg = g + (size_t)kd * nn;
    double* wr = dg + (size_t)kd * nn;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < nn * kd) {
        const int k = e / nn, m = e - k * nn;
        const double al = (k == kd - 1) ? xc + d.xb : (double)k * h + (xc - d.xb);
        const double u = xl[n0 + m] - al, gv = exp(-d.delta * u * u);
        g[e] = gv;
        dg[e] = -2.0 * d.delta * u * gv;
    } else if (e < nn * (kd + 1)) {
        const int m = e - nn * kd;
        const double x = xl[n0 + m], w = wl[n0 + m], sw = lsd_switch(d, x, xc);
        wr[m] = w;
        wr[nn + m] = 0.5 * w * (1.0 - sw);
        wr[2 * nn + m] = w * (lsd_ven(d, x) + d.v_inf * sw);
        wr[3 * nn + m] = w * exp(0.37 * (x - xc));
    }
}

// Entry (r, c), c >= r, of the overlap and the Hamiltonian of subdomain i (one
// warp), then the kd sign weights int g_k exp(0.37 (x - x_ci)): mat[i] = overlap
// [kd][kd] | Hamiltonian [kd][kd] | sign weights [kd].
__global__ void k_lsd_local_mat(LsdDev d, const int* nbase, const double* gtab, double* mat) {
    const int i = blockIdx.y, kd = d.kd, n0 = nbase[i], nn = nbase[i + 1] - n0;
    const int it = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const double* g = gtab + lsd_tab0(n0, kd);
    const double* dg = g + (size_t)kd * nn;
    const double* wr = dg + (size_t)kd * nn;
    double* Mi = mat + (size_t)i * kd * (2 * kd + 1);
    if (it < kd * kd) {
        const int r = it / kd, c = it - r * kd;
        if (c < r) return;
        const double *gr = g + (size_t)r * nn, *gc = g + (size_t)c * nn, *dr = dg + (size_t)r * nn, *dc = dg + (size_t)c * nn;
        double s = 0.0, hh = 0.0;
        for (int m = lane; m < nn; m += 32) {
            const double gg = gr[m] * gc[m];
            s += wr[m] * gg;
            hh += wr[nn + m] * (dr[m] * dc[m]) + wr[2 * nn + m] * gg;
        }
        s = warp_sum(s);
        hh = warp_sum(hh);
        if (lane == 0) {
            Mi[r * kd + c] = Mi[c * kd + r] = s;
            Mi[kd * kd + r * kd + c] = Mi[kd * kd + c * kd + r] = hh;
        }
    } else if (it < kd * kd + kd) {
        const int k = it - kd * kd;
        double s = 0.0;
        for (int m = lane; m < nn; m += 32) s += wr[3 * nn + m] * g[(size_t)k * nn + m];
        s = warp_sum(s);
        if (lane == 0) Mi[2 * kd * kd + k] = s;
    }
}

// Cyclic Jacobi of the symmetric n x n matrix B (n even, round-robin pairs):
// a round rotates n/2 disjoint index pairs.  The 2 x 2 block of two pairs is
// transformed from both sides by one thread (and mirrored), so a round is one
// pass over the upper triangle.  The rotations themselves go to `rot`
// ([round][pair] as (c, s), at most LSD_SWEEPS sweeps); the eigenvectors are
// formed from them afterwards for the wanted columns only, a quarter of the
// FP64 work of updating all of V in every round at M = 10 of 40.  The tangent
// of the angle is an FP32 estimate (the FP64 divisions and roots would be a
// serial chain of several hundred clocks in every round): the rotation stays
// orthogonal to rounding because c = 1 / sqrt(1 + t^2) is FP64, and a rotated
// entry is left at 1e-7 of what it was, which the next sweep removes.  Sweeps
// run until the off-diagonal mass is below 1e-32 of the diagonal one.
// Returns the number of rounds.
#define LSD_SWEEPS 60
__device__ inline void lsd_round_pair(int r, int k, int n, int& p, int& q) {
    // circle method: player 0 against 1 + r mod (n-1), then symmetric pairs
    if (k == 0) {
        p = 0;
        q = 1 + (r % (n - 1));
    } else {
        p = 1 + ((r + k) % (n - 1));
        q = 1 + ((r + n - 1 - k) % (n - 1));
    }
    if (p > q) {
        const int t = p;
        p = q;
        q = t;
    }
}

__device__ int lsd_jacobi(double* B, int n, double2* rot, double* red) {
    const int tid = threadIdx.x, nt = blockDim.x, half = n / 2, nblk = half * (half + 1) / 2;
    __shared__ int s_pair[LSD_KD_MAX / 2][2];
    __shared__ double s_cs[LSD_KD_MAX / 2][2];
    __shared__ int s_go;
    int rounds = 0;
    for (int sweep = 0; sweep < LSD_SWEEPS; ++sweep) {
        for (int r = 0; r < n - 1; ++r, ++rounds) {
            if (tid < half) {
                int p, q;
                lsd_round_pair(r, tid, n, p, q);
                const double apq = B[p * n + q];
                const float th = (float)(B[q * n + q] - B[p * n + p]) / (float)(2.0 * apq);
                // no rotation where the entry is zero (in FP32: negligible) or the angle is
                const float t = fabsf(th) < 1e18f ? copysignf(1.0f, th) / (fabsf(th) + sqrtf(th * th + 1.0f)) : 0.0f;
                const double td = (double)t, c = rsqrt(1.0 + td * td);
                s_pair[tid][0] = p;
                s_pair[tid][1] = q;
                s_cs[tid][0] = c;
                s_cs[tid][1] = td * c;
                rot[(size_t)rounds * half + tid] = make_double2(c, td * c);
            }
            __syncthreads();
            for (int e = tid; e < nblk; e += nt) {
                // block (k1, k2), k1 <= k2, of the triangle in row order
                int k2 = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
                while (k2 * (k2 + 1) / 2 > e) --k2;
                while ((k2 + 1) * (k2 + 2) / 2 <= e) ++k2;
                const int k1 = e - k2 * (k2 + 1) / 2;
                const int p1 = s_pair[k1][0], q1 = s_pair[k1][1], p2 = s_pair[k2][0], q2 = s_pair[k2][1];
                const double c1 = s_cs[k1][0], s1 = s_cs[k1][1], c2 = s_cs[k2][0], s2 = s_cs[k2][1];
                const double a = B[p1 * n + p2], b = B[p1 * n + q2], c = B[q1 * n + p2], dd = B[q1 * n + q2];
                const double ra = c1 * a - s1 * c, rb = c1 * b - s1 * dd, rc = s1 * a + c1 * c, rd = s1 * b + c1 * dd;
                const double oa = c2 * ra - s2 * rb, ob = s2 * ra + c2 * rb, oc = c2 * rc - s2 * rd, od = s2 * rc + c2 * rd;
                B[p1 * n + p2] = B[p2 * n + p1] = oa;
                B[q1 * n + q2] = B[q2 * n + q1] = od;
                if (k1 == k2) {
                    B[p1 * n + q1] = B[q1 * n + p1] = 0.5 * (ob + oc);
                } else {
                    B[p1 * n + q2] = B[q2 * n + p1] = ob;
                    B[q1 * n + p2] = B[p2 * n + q1] = oc;
                }
            }
            __syncthreads();
        }
        // off-diagonal mass against the diagonal (fixed-order reduction)
        double off = 0.0, dia = 0.0;
        for (int e = tid; e < n * n; e += nt) {
            const int rr = e / n, cc = e - rr * n;
            if (rr == cc) dia += B[e] * B[e];
            else off += B[e] * B[e];
        }
        off = warp_sum(off);
        dia = warp_sum(dia);
        if ((tid & 31) == 0) {
            red[tid >> 5] = off;
            red[32 + (tid >> 5)] = dia;
        }
        __syncthreads();
        if (tid == 0) {
            double o = 0.0, dsum = 0.0;
            for (int k = 0; k < nt / 32; ++k) {
                o += red[k];
                dsum += red[32 + k];
            }
            s_go = o > 1e-32 * dsum;
        }
        __syncthreads();
        if (!s_go) break;
    }
    return rounds;
}

// Eigenproblem of one subdomain: Cholesky of the overlap, L^-1 H L^-T, Jacobi,
// the M lowest eigenvectors, back substitution and the sign.  Shared memory:
// A (overlap, then its factor in the lower triangle) | B (Hamiltonian, then
// L^-1 H L^-T) | V (scratch, then the wanted eigenvectors) | W (scratch), each
// n x n with n = kd rounded up to even; the padded index is decoupled (zero
// off-diagonal entries, so no rotation touches it) and not ranked.
__global__ void __launch_bounds__(256) k_lsd_local(LsdDev d, const double* mat, double2* rot_all, double* lam_out,
                                                   double* coef_out, int* err) {
    extern __shared__ double lsm[];
    const int i = blockIdx.x, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int kd = d.kd, n = (kd + 1) & ~1, half = n / 2;
    double* A = lsm;
    double* B = A + n * n;
    double* V = B + n * n;
    double* W = V + n * n;
    double* red = W + n * n;  // 64
    __shared__ int s_ord[LSD_KD_MAX];
    __shared__ double s_inv[LSD_KD_MAX];  // 1 / L_jj
    const double* Mi = mat + (size_t)i * kd * (2 * kd + 1);
    double2* rot = rot_all + (size_t)i * LSD_SWEEPS * (n - 1) * half;
    for (int e = tid; e < n * n; e += nt) {
        const int r = e / n, c = e - r * n;
        const bool in = r < kd && c < kd;
        A[e] = in ? Mi[r * kd + c] : (r == c ? 1.0 : 0.0);
        B[e] = in ? Mi[kd * kd + r * kd + c] : 0.0;
    }
    __syncthreads();
    // Cholesky A = L L^T (right-looking, lower triangle of A)
    for (int j = 0; j < n; ++j) {
        double ljj = 1.0;
        if (j + tid < n) {  // only the warps that hold rows take the FP64 root and division
            double s = A[j * n + j];
            if (!(s > 0.0)) {
                if (tid == 0) atomicOr(err, 1);
                s = 1e-300;
            }
            ljj = sqrt(s);
        }
        __syncthreads();  // the pivot has been read
        if (j + tid < n) {
            const int r = j + tid;
            A[r * n + j] = r == j ? ljj : A[r * n + j] / ljj;
            if (r == j) s_inv[j] = 1.0 / ljj;
        }
        __syncthreads();
        const int m = n - j - 1;
        for (int e = tid; e < m * m; e += nt) {
            const int r = j + 1 + e / m, c = j + 1 + e % m;
            if (c <= r) A[r * n + c] -= A[r * n + j] * A[c * n + j];
        }
        __syncthreads();
    }
    // W = L^-1 B, then V = L^-1 W^T, right-looking row by row
    for (int pass = 0; pass < 2; ++pass) {
        double* X = pass == 0 ? W : V;
        for (int e = tid; e < n * n; e += nt) X[e] = pass == 0 ? B[e] : W[(e % n) * n + e / n];
        __syncthreads();
        for (int r = 0; r < n; ++r) {
            if (tid < n) X[r * n + tid] *= s_inv[r];
            __syncthreads();
            for (int e = tid; e < (n - r - 1) * n; e += nt) {
                const int k = r + 1 + e / n, c = e % n;
                X[k * n + c] -= A[k * n + r] * X[r * n + c];
            }
            __syncthreads();
        }
    }
    for (int e = tid; e < n * n; e += nt) {
        const int r = e / n, c = e - r * n;
        B[e] = 0.5 * (V[r * n + c] + V[c * n + r]);
    }
    __syncthreads();
    const int rounds = lsd_jacobi(B, n, rot, red);
    // ascending order of the eigenvalues (ties by index)
    if (tid < kd) {
        const double lv = B[tid * n + tid];
        int rank = 0;
        for (int k = 0; k < kd; ++k) {
            const double lk = B[k * n + k];
            rank += (lk < lv || (lk == lv && k < tid)) ? 1 : 0;
        }
        s_ord[rank] = tid;
    }
    __syncthreads();
    // the wanted columns of V = J_1 J_2 ... J_R: the rotations applied in reverse
    // to the unit vectors, one warp per column (lanes over the pairs of a round)
    for (int l = warp; l < d.M; l += nw) {
        double* v = V + l * n;
        for (int k = lane; k < n; k += 32) v[k] = k == s_ord[l] ? 1.0 : 0.0;
        __syncwarp();
        for (int t0 = rounds; t0 > 0; t0 -= 4) {
            double2 cs[4];  // the next four rounds' rotations in flight together
#pragma unroll
            for (int u = 0; u < 4; ++u)
                cs[u] = t0 - 1 - u >= 0 && lane < half ? rot[(size_t)(t0 - 1 - u) * half + lane] : make_double2(1.0, 0.0);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = t0 - 1 - u;
                if (t < 0) break;
                if (lane < half) {
                    int p, q;
                    lsd_round_pair(t % (n - 1), lane, n, p, q);
                    const double vp = v[p], vq = v[q];
                    v[p] = cs[u].x * vp + cs[u].y * vq;
                    v[q] = cs[u].x * vq - cs[u].y * vp;
                }
                __syncwarp();
            }
        }
        // X = L^-T v (back substitution, right-looking), then the sign
        for (int r = n - 1; r >= 0; --r) {
            const double x = v[r] * s_inv[r];
            __syncwarp();
            for (int k = lane; k <= r; k += 32) v[k] = k == r ? x : v[k] - A[r * n + k] * x;
            __syncwarp();
        }
        double pr = 0.0;
        for (int k = lane; k < kd; k += 32) pr += v[k] * Mi[2 * kd * kd + k];
        pr = warp_sum(pr);
        const double sg = pr < 0.0 ? -1.0 : 1.0;  // int phi exp(0.37 (x - xc)) dx > 0
        for (int k = lane; k < kd; k += 32) coef_out[((size_t)i * kd + k) * d.M + l] = sg * v[k];
        if (lane == 0) lam_out[i * d.M + l] = B[s_ord[l] * n + s_ord[l]];
    }
}

// ------------------------------------------- 2. orbitals on the global rule
// Gaussians of subdomain i at global node m (row k: [i][k][ng], values then
// derivatives) and, in row L kd, w V_en: shared by the M orbitals of i.
__global__ void k_lsd_gauss(LsdDev d, const double* xg, const double* wg, double* G, double* dG, double* wv) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x, row = blockIdx.y, kd = d.kd;
    if (m >= d.ng) return;
    const double x = xg[m];
    if (row == d.L * kd) {
        wv[m] = wg[m] * lsd_ven(d, x);
        return;
    }
    const int i = row / kd, k = row - i * kd;
    const double xc = lsd_centre(d, i), h = 2.0 * d.xb / (kd - 1);
    const double al = (k == kd - 1) ? xc + d.xb : (double)k * h + (xc - d.xb);
    const double u = x - al, gv = exp(-d.delta * u * u);
    G[(size_t)row * d.ng + m] = gv;
    dG[(size_t)row * d.ng + m] = -2.0 * d.delta * u * gv;
}

__global__ void k_lsd_table(LsdDev d, const double* G, const double* dG, const double* coef, double* F, double* dF) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x, o = blockIdx.y;
    if (m >= d.ng) return;
    const int i = o / d.M, l = o - i * d.M, kd = d.kd;
    double v = 0.0, dv = 0.0;
#pragma unroll 4
    for (int k = 0; k < kd; ++k) {
        const double c = coef[((size_t)i * kd + k) * d.M + l];
        v += c * G[((size_t)i * kd + k) * d.ng + m];
        dv += c * dG[((size_t)i * kd + k) * d.ng + m];
    }
    F[(size_t)o * d.ng + m] = v;
    dF[(size_t)o * d.ng + m] = dv;
}

// One warp per orbital pair (a, b), b >= a: overlap, one-electron Hamiltonian, position.
__global__ void k_lsd_one(LsdDev d, const double* xg, const double* wg, const double* wv, const double* F,
                          const double* dF, double* S1, double* h1, double* J1) {
    const int LM = d.L * d.M;
    const int pr = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (pr >= LM * LM) return;
    const int a = pr / LM, b = pr - a * LM;
    if (b < a) return;
    const double* fa = F + (size_t)a * d.ng;
    const double* fb = F + (size_t)b * d.ng;
    const double* da = dF + (size_t)a * d.ng;
    const double* db = dF + (size_t)b * d.ng;
    double s = 0.0, hh = 0.0, jj = 0.0;
    for (int m = lane; m < d.ng; m += 32) {
        const double pf = fa[m] * fb[m], ff = wg[m] * pf;
        s += ff;
        hh += 0.5 * wg[m] * (da[m] * db[m]) + wv[m] * pf;
        jj += xg[m] * ff;
    }
    s = warp_sum(s);
    hh = warp_sum(hh);
    jj = warp_sum(jj);
    if (lane == 0) {
        S1[pr] = S1[b * LM + a] = s;
        h1[pr] = h1[b * LM + a] = hh;
        J1[pr] = J1[b * LM + a] = jj;
    }
}

// ------------------------------------------------- 3. two-electron integrals
// Pair densities P[k][m] = w_m phi_a(x_m) phi_c(x_m) of the listed pairs.
__global__ void k_lsd_pairs(LsdDev d, const double* wg, const double* F, const int* pa, const int* pc, double* P) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (m >= d.ng) return;
    P[(size_t)k * d.ng + m] = wg[m] * F[(size_t)pa[k] * d.ng + m] * F[(size_t)pc[k] * d.ng + m];
}

// The soft-Coulomb kernel on the global nodes, W[m][s] = c / sqrt((x_m - x_s)^2 + eta^2).
__global__ void k_lsd_w(LsdDev d, const double* xg, double* Wm) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x, m = blockIdx.y;
    if (s >= d.ng) return;
    const double u = xg[m] - xg[s];
    Wm[(size_t)m * d.ng + s] = d.ee_coef / sqrt(u * u + d.eta_ee * d.eta_ee);
}

// T[k][s] = sum_m P[k][m] W[m][s] over the pair's support nodes [lo, hi)
// (rows of W read along s: coalesced; P staged in shared memory).
__global__ void k_lsd_pw(LsdDev d, const double* Wm, const double* P, const int* lo, const int* hi, double* T) {
    __shared__ double sp[256];
    const int k = blockIdx.y, s = blockIdx.x * blockDim.x + threadIdx.x;
    double acc = 0.0;
    for (int m0 = lo[k]; m0 < hi[k]; m0 += 256) {
        const int m = m0 + threadIdx.x;
        sp[threadIdx.x] = m < hi[k] ? P[(size_t)k * d.ng + m] : 0.0;
        __syncthreads();
        const int cnt = min(256, hi[k] - m0);
        if (s < d.ng)
            for (int j = 0; j < cnt; ++j) acc += sp[j] * Wm[(size_t)(m0 + j) * d.ng + s];
        __syncthreads();
    }
    if (s < d.ng) T[(size_t)k * d.ng + s] = acc;
}

// ----------------------------------------------- 4. determinants per Omega
// Rank of every candidate (l, p) of Omega_{i,j} (i = om mod L, j = om / L) by
// lambda_l^i + lambda_p^j with the tie rule; the first K kept.
__global__ void k_lsd_select(LsdDev d, const double* lam, int* pairs, int* err) {
    const int om = blockIdx.x, i = om % d.L, j = om / d.L, M = d.M;
    const int nc = (i == j) ? M * (M - 1) / 2 : M * M;
    for (int u = threadIdx.x; u < nc; u += blockDim.x) {
        // candidate u: (l, p) in lexicographic order among the allowed pairs
        auto cand = [&](int v, int& l, int& p) {
            if (i != j) {
                l = v / M;
                p = v - l * M;
            } else {
                l = 0;
                int rem = v;
                while (rem >= M - 1 - l) {
                    rem -= M - 1 - l;
                    ++l;
                }
                p = l + 1 + rem;
            }
        };
        int lu, pu;
        cand(u, lu, pu);
        const double eu = lam[i * M + lu] + lam[j * M + pu];
        int rank = 0;
        for (int v = 0; v < nc; ++v) {
            if (v == u) continue;
            int lv, pv;
            cand(v, lv, pv);
            const double ev = lam[i * M + lv] + lam[j * M + pv], df = ev - eu;
            bool before;
            if (fabs(df) <= LSD_TIE * (1.0 + fabs(eu) + fabs(ev))) before = (lv < lu) || (lv == lu && pv < pu);
            else before = df < 0.0;
            rank += before ? 1 : 0;
        }
        if (rank < d.K) {
            int* q = pairs + ((size_t)om * d.K + rank) * 2;
            if (atomicCAS(q, -1, lu) != -1) atomicOr(err, 2);  // two candidates on one rank
            q[1] = pu;
        }
    }
}

// Gram, H0 and the Gram against Omega_{i+1,j}: one warp per entry (r, c).
__global__ void k_lsd_blocks(LsdDev d, const int* pairs, const double* S1, const double* h1, const double* T,
                             const double* P, const int* pid, const int* lo, const int* hi, double* S_lsd,
                             double* H_lsd, double* G_next) {
    const int om = blockIdx.y, i = om % d.L, j = om / d.L, M = d.M, K = d.K, LM = d.L * d.M;
    const int e = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (e >= K * K) return;
    const int r = e / K, c = e - r * K;
    const int* pr = pairs + ((size_t)om * K + r) * 2;
    const int* pc = pairs + ((size_t)om * K + c) * 2;
    // a rank left empty by the selection (reported there): no index to read
    if (pr[0] < 0 || pr[1] < 0 || pc[0] < 0 || pc[1] < 0 ||
        (i + 1 < d.L && (pairs[((size_t)(om + 1) * K + c) * 2] < 0 || pairs[((size_t)(om + 1) * K + c) * 2 + 1] < 0))) {
        if (lane == 0) {
            const size_t o = (size_t)om * K * K + e;
            S_lsd[o] = H_lsd[o] = G_next[o] = nan("");
        }
        return;
    }
    const int a = i * M + pr[0], b = j * M + pr[1], cc = i * M + pc[0], dd = j * M + pc[1];
    const double sac = S1[a * LM + cc], sbd = S1[b * LM + dd], sad = S1[a * LM + dd], sbc = S1[b * LM + cc];
    // (xy|zw) = T_{xy} . P_{zw} over the support of the pair zw; 0 when a pair's
    // supports are disjoint (no pair density listed)
    auto eri = [&](int x, int y, int z, int w) -> double {
        const int k1 = pid[x * LM + y], k2 = pid[z * LM + w];
        double s = 0.0;
        if (k1 >= 0 && k2 >= 0)
            for (int m = lo[k2] + lane; m < hi[k2]; m += 32) s += T[(size_t)k1 * d.ng + m] * P[(size_t)k2 * d.ng + m];
        return warp_sum(s);
    };
    const double one = h1[a * LM + cc] * sbd + sac * h1[b * LM + dd] - h1[a * LM + dd] * sbc - sad * h1[b * LM + cc];
    const double two = eri(a, cc, b, dd) - eri(a, dd, b, cc);
    double gn = 0.0;
    if (i + 1 < d.L) {
        const int* pn = pairs + ((size_t)(om + 1) * K + c) * 2;  // Omega_{i+1,j}
        const int c2 = (i + 1) * M + pn[0], d2 = j * M + pn[1];
        gn = S1[a * LM + c2] * S1[b * LM + d2] - S1[a * LM + d2] * S1[b * LM + c2];
    }
    if (lane == 0) {
        const size_t o = (size_t)om * K * K + e;
        S_lsd[o] = sac * sbd - sad * sbc;
        H_lsd[o] = one + two;
        G_next[o] = gn;
    }
}

}  // namespace swr

// ------------------------------------------------------------- host side
using namespace swr;

namespace {
std::string g_lsd_err;

swr_status lsd_fail(swr_status s, const char* msg) {
    g_lsd_err = msg;
    set_setup_error(msg);
    return s;
}

// Composite rule panels on [lo, hi] with edges at the breakpoints inside and
// panels of width <= panel between them (k step + s0, the last edge exact).
void lsd_panels(double lo, double hi, double panel, const std::vector<double>& brk, std::vector<double>& edges,
                std::vector<int>& ebase) {
    std::vector<double> pts = {lo, hi};
    for (double b : brk)
        if (b > lo && b < hi) pts.push_back(b);
    std::sort(pts.begin(), pts.end());
    pts.erase(std::unique(pts.begin(), pts.end()), pts.end());
    for (size_t s = 0; s + 1 < pts.size(); ++s) {
        const double s0 = pts[s], s1 = pts[s + 1];
        int n = (int)ceil((s1 - s0) / panel - 1e-12);
        if (n < 1) n = 1;
        const double step = (s1 - s0) / n;
        const size_t first = edges.size();
        for (int k = 0; k < n; ++k) edges.push_back(k == 0 ? s0 : (double)k * step + s0);
        edges.push_back(s1);
        for (int k = 0; k < n; ++k) ebase.push_back((int)(first + k));
    }
}

// Device memory of one call: pieces of one allocation, 256-byte aligned.
struct DevBuf {
    char* base = nullptr;
    size_t used = 0;
    ~DevBuf() { cudaFree(base); }
    template <class T>
    size_t add(size_t n) {
        const size_t o = used;
        used += ((n ? n : 1) * sizeof(T) + 255) & ~(size_t)255;
        return o;
    }
    template <class T>
    T* at(size_t o) const { return reinterpret_cast<T*>(base + o); }
};
}  // namespace

extern "C" swr_status swr_lsd_build(const swr_lsd_problem* p, swr_lsd_result* out) {
    if (!p || !out) return lsd_fail(SWR_EINVAL, "swr_lsd_build: problem or result is NULL");
    if (!out->lam || !out->coef || !out->S1 || !out->h1 || !out->J1 || !out->pairs || !out->S_lsd || !out->H_lsd ||
        !out->G_next)
        return lsd_fail(SWR_EINVAL, "swr_lsd_build: every result buffer must be given");
    if (!(p->box_hi > p->box_lo) || p->L < 1 || p->L > 16 || !(p->overlap >= 0.0))
        return lsd_fail(SWR_EINVAL, "swr_lsd_build: need box_lo < box_hi, 1 <= L <= 16, overlap >= 0");
    if (p->kd < 2 || p->kd > LSD_KD_MAX || p->M < 1 || p->M > p->kd)
        return lsd_fail(SWR_EINVAL, "swr_lsd_build: need 2 <= kd <= 64 and 1 <= M <= kd");
    if (p->K < 1 || p->K > p->M * (p->M - 1) / 2)
        return lsd_fail(SWR_EINVAL, "swr_lsd_build: need 1 <= K <= M (M - 1) / 2 (determinants of a diagonal subdomain)");
    if (p->q_p < 2 || p->q_p > LSD_Q_MAX || !(p->panel > 0.0))
        return lsd_fail(SWR_EINVAL, "swr_lsd_build: need 2 <= q_p <= 16 and panel > 0");
    if (p->n_nuclei < 0 || p->n_nuclei > 3 || (p->n_nuclei > 0 && !(p->eta_en > 0.0)) || !(p->eta_ee > 0.0))
        return lsd_fail(SWR_EINVAL, "swr_lsd_build: at most 3 nuclei; eta_en > 0 with nuclei; eta_ee > 0");
    if (!(p->xb_factor > 0.0) || !(p->eps_b > 0.0) || !(p->v_inf >= 0.0) || !(p->delta >= 0.0))
        return lsd_fail(SWR_EINVAL, "swr_lsd_build: need xb_factor > 0, eps_b > 0, v_inf >= 0, delta >= 0");
    LsdDev d;
    memset(&d, 0, sizeof(d));
    d.L = p->L;
    d.M = p->M;
    d.K = p->K;
    d.kd = p->kd;
    d.q = p->q_p;
    d.a = p->box_lo;
    d.H = (p->box_hi - p->box_lo) / p->L;
    d.eps = p->overlap;
    const double width = d.H + d.eps;  // |D_i|
    d.xb = p->xb_factor * width;
    d.eps_b = p->eps_b;
    d.v_inf = p->v_inf;
    const double hc = 2.0 * d.xb / (p->kd - 1);
    d.delta = p->delta > 0.0 ? p->delta : 0.5 / (hc * hc);
    d.eta_en = p->eta_en;
    d.eta_ee = p->eta_ee;
    d.ee_coef = p->ee_coef;
    d.harmonic = p->harmonic;
    d.n_nuc = p->n_nuclei;
    for (int A = 0; A < p->n_nuclei; ++A) {
        d.xn[A] = p->x_nuc[A];
        d.zn[A] = p->Z_nuc[A];
    }
    const double margin = std::max(p->eps_b, 8.0 / sqrt(2.0 * d.delta));
    // local rules (breakpoints where the barrier's step starts and ends) and the global rule
    std::vector<double> edges;
    std::vector<int> ebase, nbase = {0};
    for (int i = 0; i < p->L; ++i) {
        const double xc = d.a + (i + 0.5) * d.H, e = 0.5 * p->eps_b;
        const size_t before = ebase.size();
        lsd_panels(xc - d.xb - margin, xc + d.xb + margin, p->panel,
                   {xc - d.xb - e, xc - d.xb + e, xc + d.xb - e, xc + d.xb + e}, edges, ebase);
        nbase.push_back(nbase.back() + (int)(ebase.size() - before) * p->q_p);
    }
    const int n_local_panels = (int)ebase.size();
    const double gm = d.xb - 0.5 * width + margin;
    const double glo = p->box_lo - 0.5 * p->overlap - gm, ghi = p->box_hi + 0.5 * p->overlap + gm;
    lsd_panels(glo, ghi, p->panel, {}, edges, ebase);
    const int n_global_panels = (int)ebase.size() - n_local_panels;
    d.ng = n_global_panels * p->q_p;
    const int LM = p->L * p->M, nloc = nbase.back();
    // pair densities of orbitals in the same or neighbouring subdomains, with the
    // node range where both are above the Gaussian tails
    std::vector<int> pa, pc, plo, phi, pid(LM * LM, -1);
    auto node_of = [&](double x) {  // first global node at or after x
        const double pw = (ghi - glo) / n_global_panels;
        int pnl = (int)floor((x - glo) / pw);
        pnl = std::min(std::max(pnl, 0), n_global_panels);
        return pnl * p->q_p;
    };
    for (int a = 0; a < LM; ++a)
        for (int c = a; c < LM; ++c) {
            const int ia = a / p->M, ic = c / p->M;
            const double xa = d.a + (ia + 0.5) * d.H, xc2 = d.a + (ic + 0.5) * d.H;
            const double lo = std::max(xa, xc2) - d.xb - margin, hi = std::min(xa, xc2) + d.xb + margin;
            if (!(hi > lo)) continue;  // supports (x_ci -+ (x_b + margin)) apart
            pid[a * LM + c] = pid[c * LM + a] = (int)pa.size();
            pa.push_back(a);
            pc.push_back(c);
            plo.push_back(node_of(lo));
            phi.push_back(std::min(d.ng, node_of(hi) + p->q_p));
        }
    d.n_pairs = (int)pa.size();
    if (d.n_pairs > 65535) return lsd_fail(SWR_EINVAL, "swr_lsd_build: more than 65535 orbital pairs (L M too large)");
    // device work: the host tables packed into one upload, the results into one
    // read-back (an allocation and a copy for each array cost a millisecond)
    DevBuf db;
    const int n = (p->kd + 1) & ~1, np = n_local_panels + n_global_panels;
    const size_t nblk = (size_t)p->L * p->L * p->K * p->K;
    const size_t o_edges = db.add<double>(edges.size()), o_ebase = db.add<int>(ebase.size()),
                 o_nbase = db.add<int>(nbase.size()), o_pa = db.add<int>(pa.size()), o_pc = db.add<int>(pc.size()),
                 o_lo = db.add<int>(plo.size()), o_hi = db.add<int>(phi.size()), o_pid = db.add<int>(pid.size()),
                 up_bytes = db.used;
    const size_t o_lam = db.add<double>(LM), o_coef = db.add<double>((size_t)p->L * p->kd * p->M),
                 o_S1 = db.add<double>((size_t)LM * LM), o_h1 = db.add<double>((size_t)LM * LM),
                 o_J1 = db.add<double>((size_t)LM * LM), o_pairs = db.add<int>((size_t)p->L * p->L * p->K * 2),
                 o_Sl = db.add<double>(nblk), o_Hl = db.add<double>(nblk), o_Gn = db.add<double>(nblk),
                 o_err = db.add<int>(1), down_end = db.used;
    const size_t o_t = db.add<double>(LSD_Q_MAX), o_w = db.add<double>(LSD_Q_MAX),
                 o_x = db.add<double>((size_t)(nloc + d.ng)), o_wx = db.add<double>((size_t)(nloc + d.ng)),
                 o_gtab = db.add<double>(lsd_tab0(nloc, p->kd)),
                 o_mat = db.add<double>((size_t)p->L * p->kd * (2 * p->kd + 1)),
                 o_rot = db.add<double2>((size_t)p->L * LSD_SWEEPS * (n - 1) * (n / 2)),
                 o_G = db.add<double>((size_t)p->L * p->kd * d.ng), o_dG = db.add<double>((size_t)p->L * p->kd * d.ng),
                 o_wv = db.add<double>(d.ng), o_F = db.add<double>((size_t)LM * d.ng),
                 o_dF = db.add<double>((size_t)LM * d.ng), o_P = db.add<double>((size_t)d.n_pairs * d.ng),
                 o_T = db.add<double>((size_t)d.n_pairs * d.ng), o_W = db.add<double>((size_t)d.ng * d.ng);
    if (cudaMalloc((void**)&db.base, db.used) != cudaSuccess) {
        db.base = nullptr;
        cudaGetLastError();
        return lsd_fail(SWR_ENOMEM, "swr_lsd_build: device allocation failed");
    }
    std::vector<char> hbuf(std::max(up_bytes, down_end - up_bytes));
    auto pack = [&](size_t o, const void* src, size_t bytes) { memcpy(hbuf.data() + o, src, bytes); };
    pack(o_edges, edges.data(), edges.size() * sizeof(double));
    pack(o_ebase, ebase.data(), ebase.size() * sizeof(int));
    pack(o_nbase, nbase.data(), nbase.size() * sizeof(int));
    pack(o_pa, pa.data(), pa.size() * sizeof(int));
    pack(o_pc, pc.data(), pc.size() * sizeof(int));
    pack(o_lo, plo.data(), plo.size() * sizeof(int));
    pack(o_hi, phi.data(), phi.size() * sizeof(int));
    pack(o_pid, pid.data(), pid.size() * sizeof(int));
    double *dt = db.at<double>(o_t), *dw = db.at<double>(o_w), *dx = db.at<double>(o_x), *dwx = db.at<double>(o_wx);
    double *dlam = db.at<double>(o_lam), *dcoef = db.at<double>(o_coef), *dF = db.at<double>(o_F), *ddF = db.at<double>(o_dF);
    double *dS1 = db.at<double>(o_S1), *dh1 = db.at<double>(o_h1), *dJ1 = db.at<double>(o_J1);
    double *dP = db.at<double>(o_P), *dT = db.at<double>(o_T), *dWm = db.at<double>(o_W);
    const int *dnbase = db.at<int>(o_nbase), *dplo = db.at<int>(o_lo), *dphi = db.at<int>(o_hi), *dpid = db.at<int>(o_pid);
    int *dpairs = db.at<int>(o_pairs), *derr = db.at<int>(o_err);
    cudaError_t e = cudaSuccess;
#define LSD_CU(call)                                                               \
    do {                                                                           \
        if (e == cudaSuccess) e = (call);                                          \
    } while (0)
    LSD_CU(cudaMemcpy(db.base, hbuf.data(), up_bytes, cudaMemcpyHostToDevice));
    LSD_CU(cudaMemsetAsync(dpairs, 0xff, (size_t)p->L * p->L * p->K * 2 * sizeof(int)));
    LSD_CU(cudaMemsetAsync(derr, 0, sizeof(int)));
    if (e == cudaSuccess) {
        int nn_max = 0;
        for (int i = 0; i < p->L; ++i) nn_max = std::max(nn_max, nbase[i + 1] - nbase[i]);
        k_lsd_gl<<<1, LSD_Q_MAX>>>(p->q_p, dt, dw);
        const int nn = np * p->q_p;
        k_lsd_nodes<<<(nn + 255) / 256, 256>>>(db.at<double>(o_edges), db.at<int>(o_ebase), np, dt, dw, p->q_p, dx, dwx);
        const int nt = 256;
        const size_t smem = (4 * (size_t)n * n + 64) * sizeof(double);
        LSD_CU(allow_dynamic_smem((const void*)k_lsd_local));
        k_lsd_local_tab<<<dim3((nn_max * (p->kd + 1) + 255) / 256, p->L), 256>>>(d, dx, dwx, dnbase, db.at<double>(o_gtab));
        k_lsd_local_mat<<<dim3((p->kd * (p->kd + 1) + 7) / 8, p->L), 256>>>(d, dnbase, db.at<double>(o_gtab),
                                                                           db.at<double>(o_mat));
        k_lsd_local<<<p->L, nt, smem>>>(d, db.at<double>(o_mat), db.at<double2>(o_rot), dlam, dcoef, derr);
        const double* xg = dx + nloc;
        const double* wg = dwx + nloc;
        k_lsd_gauss<<<dim3((d.ng + 127) / 128, p->L * p->kd + 1), 128>>>(d, xg, wg, db.at<double>(o_G), db.at<double>(o_dG),
                                                                       db.at<double>(o_wv));
        k_lsd_table<<<dim3((d.ng + 127) / 128, LM), 128>>>(d, db.at<double>(o_G), db.at<double>(o_dG), dcoef, dF, ddF);
        k_lsd_one<<<(LM * LM + 7) / 8, 256>>>(d, xg, wg, db.at<double>(o_wv), dF, ddF, dS1, dh1, dJ1);
        k_lsd_pairs<<<dim3((d.ng + 255) / 256, d.n_pairs), 256>>>(d, wg, dF, db.at<int>(o_pa), db.at<int>(o_pc), dP);
        k_lsd_w<<<dim3((d.ng + 255) / 256, d.ng), 256>>>(d, xg, dWm);
        k_lsd_pw<<<dim3((d.ng + 255) / 256, d.n_pairs), 256>>>(d, dWm, dP, dplo, dphi, dT);
        k_lsd_select<<<p->L * p->L, 256>>>(d, dlam, dpairs, derr);
        k_lsd_blocks<<<dim3((p->K * p->K + 7) / 8, p->L * p->L), 256>>>(d, dpairs, dS1, dh1, dT, dP, dpid, dplo, dphi,
                                                                       db.at<double>(o_Sl), db.at<double>(o_Hl),
                                                                       db.at<double>(o_Gn));
        LSD_CU(cudaGetLastError());
    }
    int herr = 0;
    LSD_CU(cudaMemcpy(hbuf.data(), db.base + up_bytes, down_end - up_bytes, cudaMemcpyDeviceToHost));
    if (e == cudaSuccess) {
        auto take = [&](void* dst, size_t o, size_t bytes) { memcpy(dst, hbuf.data() + (o - up_bytes), bytes); };
        take(&herr, o_err, sizeof(int));
        take(out->lam, o_lam, (size_t)LM * sizeof(double));
        take(out->coef, o_coef, (size_t)p->L * p->kd * p->M * sizeof(double));
        take(out->S1, o_S1, (size_t)LM * LM * sizeof(double));
        take(out->h1, o_h1, (size_t)LM * LM * sizeof(double));
        take(out->J1, o_J1, (size_t)LM * LM * sizeof(double));
        take(out->pairs, o_pairs, (size_t)p->L * p->L * p->K * 2 * sizeof(int));
        take(out->S_lsd, o_Sl, nblk * sizeof(double));
        take(out->H_lsd, o_Hl, nblk * sizeof(double));
        take(out->G_next, o_Gn, nblk * sizeof(double));
    }
#undef LSD_CU
    if (e != cudaSuccess) {
        char msg[256];
        snprintf(msg, sizeof(msg), "swr_lsd_build: %s", cudaGetErrorString(e));
        return lsd_fail(SWR_ECUDA, msg);
    }
    if (herr & 1) return lsd_fail(SWR_ESINGULAR, "swr_lsd_build: an orbital basis overlap is not positive definite");
    if (herr & 2) return lsd_fail(SWR_ENUMERIC, "swr_lsd_build: the tie rule does not order the determinants");
    return SWR_OK;
}
