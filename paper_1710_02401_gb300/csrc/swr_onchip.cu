// swr_onchip.cu -- the FP64 imaginary-time window of small instances, one
// thread-block cluster per instance.
//
// The recursion of the two-phase window (swr_window.cu):
//     y^{n+1} = G v^n,  v^n = y^n / s_n + kappa dt b'^{n+1},
//     s_n^2 = sum_i y_i^n . z_i^n,  z = (Pp (x) Pp) y,
// with its stops (first n >= 1 with ||c^n - c^{n-1}|| <= tol, the cap, or a
// normalisation that is not positive and finite).  Small problems are bound by
// the latency of a step: 2 subdomains of 40 Gaussians took 15.6 us a step in
// the two-phase kernel, two grid barriers through L2 and FP64 chains (66 clocks
// an addition) over a handful of CTAs; 2.9 us here (9 subdomains of K = 121: 16.0
// -> 6.0), still latency: the cluster barrier, the FP64 sums of the
// partials and the reciprocal root follow one another.  The whole instance
// sits in the shared memory of one cluster:
//  - the rows of all its subdomains are dealt to the CTAs by matrix elements;
//  - with W = (Pp (x) Pp) G (formed at assembly in the space of H', which is not
//    needed any more) z^{n+1} = W v^n comes out of the same pass as y^{n+1}, so a
//    step has one barrier, and that is the cluster's;
//  - y rows go to the CTAs of their subdomain and the partials of s^2 and of the
//    stop test to every CTA through distributed shared memory;
//  - the products run in 56-bit fixed point (swr_fixed.cuh; matrix rows scaled by
//    their 2-norm.  By their largest entry with two bits kept free, the product of 40
//    rows with a smooth vector was 1.8e-16 off in norm, 0.8e-16 in FP64; so it is
//    0.4e-16): exact sums at 4.5 multiply-adds per clock and SM against 1.6
//    on the FP64 pipe and, what counts here, additions of 4 clocks instead of 66.
// Everything else stays FP64.
#include <math.h>

#include <vector>

#include "swr_fixed.cuh"

namespace swr {

#define OC_THREADS 512
#define OC_WARPS 16
#define OC_CMAX 16                 // CTAs per cluster (at most)
#define OC_SMEM_MAX (224 * 1024)
#define OC_KMAX 256                // K of a subdomain (at most)
#define OC_SUBS 64                 // subdomains with rows in one CTA (at most)

// Limb pairs per matrix row: an odd number of 64-byte segments (8 columns), so
// that the G and W rows of two neighbouring rows start in alternate bank halves.
__host__ __device__ inline int oc_pitch(int K) { return 8 * (((K + 7) / 8) | 1); }

__device__ inline unsigned oc_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ inline void oc_store(const void* local, unsigned rank, double x) {
    unsigned ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(oc_smem(local)), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(x) : "memory");
}
__device__ inline void oc_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

struct OcArgs {
    SwrDeviceView v;
    const int* bounds;     // [n_inst][cs + 1] first row of each CTA (rows of the instance's subdomains in order)
    const int* row0;       // [n_sub] first row of a subdomain within its instance
    const int* win_prev;
    double* snorm;
    int* win;
    int* n_active;
    int cap, cs, tune_steps, rows_max, nv_max, lim_max;
};

__host__ __device__ inline size_t oc_smem_bytes(int rows_max, int nv_max, int lim_max) {
    return (size_t)lim_max * sizeof(int2) +                       // G, W limbs
           (size_t)nv_max * (2 * sizeof(double) + sizeof(int2)) +  // y (two steps), v limbs
           (size_t)rows_max * (8 * sizeof(double) + 4 * sizeof(int)) + 64;  // y, z of three steps, products; row tables
}

// W = (Pp1 (x) Pp2) G (Pp1 G with one electron), FP64, into the space of H', one column per CTA.
__global__ void k_oc_make_w(SwrDeviceView v) {
    const SubDev& s = v.sub[blockIdx.y];
    const int K = s.K, kd = s.kd;
    T1Layout lay(s.q, kd);
    const double* P1 = v.arena + s.t1[0] + lay.mat(M_PP);
    const double* P2 = v.arena + s.t1[s.N == 2 ? 1 : 0] + lay.mat(M_PP);
    const double* G = v.arena + s.Gm;
    double* W = v.arena + s.Hm;
    __shared__ double Y[1024], T[1024];  // K <= 1024
    for (int j = blockIdx.x; j < K; j += gridDim.x) {
        for (int r = threadIdx.x; r < K; r += blockDim.x) Y[r] = G[(long long)r * K + j];
        __syncthreads();
        for (int e2 = threadIdx.x; e2 < K; e2 += blockDim.x) {  // T[a + kd e] = sum_c P1[a][c] Y[c + kd e]
            const int e = e2 / kd, a = e2 - e * kd;
            double acc = 0;
            for (int c = 0; c < kd; ++c) acc = fma(P1[a * kd + c], Y[c + kd * e], acc);
            T[e2] = acc;
        }
        __syncthreads();
        for (int m = threadIdx.x; m < K; m += blockDim.x) {
            const int b = m / kd, a = m - b * kd;
            double acc = T[m];
            if (s.N == 2) {
                acc = 0;
                for (int e = 0; e < kd; ++e) acc = fma(T[a + kd * e], P2[b * kd + e], acc);
            }
            W[(long long)m * K + j] = acc;
        }
        __syncthreads();
    }
}

// Sum of n values over a warp (fixed order), to every lane.
__device__ inline double oc_warp_total(const double* x, int n, int lane) {
    double a = 0;
    for (int i = lane; i < n; i += 32) a += x[i];
    return warp_sum(a);
}

__global__ void __launch_bounds__(OC_THREADS, 1) k_window_onchip(OcArgs A) {
    extern __shared__ __align__(16) unsigned char oc_sm[];
    __shared__ __align__(16) double2 s_slot[2][OC_CMAX];  // partials of s_n^2 and D_{n-1} by step parity and CTA
    __shared__ int s_emax[2][OC_SUBS];                    // exponent of v per subdomain here, by step parity
    __shared__ int s_base[OC_CMAX], s_bound[OC_CMAX + 1]; // first row of y kept by each CTA; its first own row
    __shared__ int s_sub0[OC_SUBS + 1];  // per subdomain here: first row
    __shared__ double s_is[2];                            // 1/s_n, 1/s_{n-1}
    __shared__ int s_stop;
    const SwrDeviceView& v = A.v;
    const int CS = A.cs, inst = blockIdx.x / CS, rank = blockIdx.x % CS;
    const InstDev& in = v.inst[inst];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int* bounds = A.bounds + (long long)inst * (CS + 1);
    const int* row0 = A.row0 + in.sub_base;
    auto sub_of = [&](int row) {  // subdomain (within the instance) of a row
        int s = 0;
        while (s + 1 < in.n_sub && row0[s + 1] <= row) ++s;
        return s;
    };
    const int r0 = bounds[rank], r1 = bounds[rank + 1], nr = r1 - r0;
    const int sA = sub_of(r0), sB = sub_of(nr > 0 ? r1 - 1 : r0), nsub = sB - sA + 1;
    const int v0 = row0[sA], nv = row0[sB] + v.sub[in.sub_base + sB].K - v0;  // rows of y needed here
    if (tid <= CS) s_bound[tid] = bounds[tid];
    if (tid < CS) s_base[tid] = row0[sub_of(bounds[tid])];
    if (tid <= nsub) s_sub0[tid] = tid < nsub ? row0[sA + tid] : v0 + nv;
    if (tid < OC_SUBS) s_emax[0][tid] = s_emax[1][tid] = 0;
    int2* lim = reinterpret_cast<int2*>(oc_sm);
    double* yf = reinterpret_cast<double*>(lim + A.lim_max);  // [2][nv_max]
    double* yo = yf + 2 * A.nv_max;                           // [3][rows_max]
    double* zo = yo + 3 * A.rows_max;                         // [3][rows_max]
    double* ps = zo + 3 * A.rows_max;                         // y^{n+1} z^{n+1} per own row
    double* pd = ps + A.rows_max;                             // terms of D_n
    int2* vl = reinterpret_cast<int2*>(pd + A.rows_max);      // [nv_max] limbs of v
    int* r_off = reinterpret_cast<int*>(vl + A.nv_max);       // [rows_max] limbs of the row (G, then W)
    int* r_sub = r_off + A.rows_max;                          // local subdomain
    int* r_eg = r_sub + A.rows_max;                           // exponents of the G and W rows
    int* r_ew = r_eg + A.rows_max;
    __syncthreads();
    // ------------------------------------------------------------- set-up
    if (tid == 0) {
        int off = 0;
        for (int i = 0, ls = 0; i < nr; ++i) {
            while (s_sub0[ls + 1] <= r0 + i) ++ls;
            r_off[i] = off;
            r_sub[i] = ls;
            off += 2 * oc_pitch(s_sub0[ls + 1] - s_sub0[ls]);
        }
    }
    __syncthreads();
    for (int i = warp; i < nr; i += OC_WARPS) {  // a warp per row: exponents and limbs of G and W
        const SubDev& s = v.sub[in.sub_base + sA + r_sub[i]];
        const int K = s.K, pitch = oc_pitch(K), r = r0 + i - s_sub0[r_sub[i]];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const double* row = v.arena + (h ? s.Hm : s.Gm) + (long long)r * K;
            int e = 0;
            for (int c = lane; c < K; c += 32) e = max(e, fx_exp(row[c]));
            e = __reduce_max_sync(0xffffffffu, e);
            const double sc = fx_row_scale(e);
            float q = 0.f;
            for (int c = lane; c < K; c += 32) {
                const float t = (float)(row[c] * sc);
                q += t * t;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
            e = fx_row_exp(e, q);
            for (int c = lane; c < pitch; c += 32) lim[r_off[i] + h * pitch + c] = c < K ? fx_limbs(row[c], e) : make_int2(0, 0);
            if (lane == 0) (h ? r_ew : r_eg)[i] = e;
        }
    }
    for (int j = tid; j < nv; j += OC_THREADS) {
        int ls = 0;
        while (s_sub0[ls + 1] <= v0 + j) ++ls;
        yf[j] = v.arena[v.sub[in.sub_base + sA + ls].c0 + (v0 + j - s_sub0[ls])];
        vl[j] = make_int2(0, 0);
    }
    __syncthreads();
    // y^0 = c0 and z^0 = (Pp (x) Pp) y^0 of the own rows
    for (int i = tid; i < nr; i += OC_THREADS) {
        const int ls = r_sub[i];
        const SubDev& s = v.sub[in.sub_base + sA + ls];
        const int kd = s.kd, r = r0 + i - s_sub0[ls], b = s.N == 2 ? r / kd : 0, a = r - b * kd;
        T1Layout lay(s.q, kd);
        const double* P1 = v.arena + s.t1[0] + lay.mat(M_PP) + a * kd;
        const double* P2 = v.arena + s.t1[s.N == 2 ? 1 : 0] + lay.mat(M_PP) + b * kd;
        const double* y = yf + (s_sub0[ls] - v0);
        double z = 0;
        for (int e = 0; e < (s.N == 2 ? kd : 1); ++e) {
            double t = 0;
            for (int c = 0; c < kd; ++c) t = fma(P1[c], y[c + kd * e], t);
            z = s.N == 2 ? fma(P2[e], t, z) : t;
        }
        yo[i] = y[r];
        zo[i] = z;
        ps[i] = y[r] * z;
        v.arena[s.hist + r] = y[r];
    }
    const int wp = A.win_prev[inst];
    int maxs = in.window_cap > 0 ? in.window_cap : in.max_steps;
    bool stop_rule = in.window_cap == 0 && in.ngf_tol > 0.0;
    if (A.tune_steps > 0) {
        maxs = min(maxs, A.tune_steps);
        stop_rule = false;
    }
    const double kdt = in.kappa * in.dt;
    // this thread's entries of v: tid, tid + 512, ... (the first one's b' is loaded a step ahead)
    auto b_of = [&](int j, int n) -> double {
        if (wp <= 0) return 0.0;
        int ls = 0;
        while (s_sub0[ls + 1] <= v0 + j) ++ls;
        const SubDev& s = v.sub[in.sub_base + sA + ls];
        return v.arena[s.bvec + (long long)min(n, wp) * s.K + (v0 + j - s_sub0[ls])];
    };
    int ls_t = 0;  // local subdomain and b' of entry tid
    const double* b_t = nullptr;
    long long bK = 0;
    if (tid < nv) {
        while (s_sub0[ls_t + 1] <= v0 + tid) ++ls_t;
        const SubDev& s = v.sub[in.sub_base + sA + ls_t];
        if (wp > 0) b_t = v.arena + s.bvec + (v0 + tid - s_sub0[ls_t]);
        bK = s.K;
    }
    double b_next = b_t ? b_t[(long long)min(1, wp) * bK] : 0.0;
    // partials to every CTA: warp 0 the s^2, warp 1 the D
    auto publish = [&](int par) {
        if (warp < 2) {
            const double t = oc_warp_total(warp ? pd : ps, nr, lane);
            if (lane < CS) {
                double2* slot = &s_slot[par][rank];
                oc_store(warp ? &slot->y : &slot->x, (unsigned)lane, t);
            }
        }
    };
    for (int i = tid; i < nr; i += OC_THREADS) pd[i] = 0.0;
    oc_sync();  // every CTA runs before the first remote store; this CTA's set-up is complete
    publish(0);
    oc_sync();

    for (int n = 0;; ++n) {
        const int par = n & 1;
        const double bv = b_next;
        // ---- s_n, D_{n-1}, the decisions of step n (the same bits in every CTA)
        if (warp == 0) {
            double s2 = lane < CS ? s_slot[par][lane].x : 0.0, d2 = lane < CS ? s_slot[par][lane].y : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                s2 += __shfl_xor_sync(0xffffffffu, s2, o);
                d2 += __shfl_xor_sync(0xffffffffu, d2, o);
            }
            if (lane == 0) {
                const double is = in.normalize ? rsqrt(s2) : 1.0, sn = in.normalize ? s2 * is : 1.0;
                const bool bad = !isfinite(sn) || !(sn > 0.0);
                int stop = 0;
                if (n >= 2 && stop_rule && d2 <= in.ngf_tol * in.ngf_tol) stop = 1;  // the window ends at n - 1
                else if (n >= maxs || bad) stop = 2;                                 // at n
                s_stop = stop;
                s_is[1] = s_is[0];
                s_is[0] = is;
                if (rank == 0) {
                    if (stop != 1) A.snorm[(long long)inst * (A.cap + 1) + n] = sn;
                    if (stop) {
                        A.win[inst] = stop == 1 ? n - 1 : n;
                        if (stop == 2 && bad) atomicOr(v.err, SWR_ERR_NUMERIC);
                        atomicSub(A.n_active, 1);
                    }
                }
            }
        }
        __syncthreads();
        if (s_stop) break;
        const double is = s_is[0], is_p = s_is[1];
        // ---- v = y^n / s_n + kappa dt b'^{n+1} and its exponent per subdomain
        const double* yn = yf + par * A.nv_max;
        double vt = 0.0;
        if (tid < nv) {
            vt = fma(kdt, bv, yn[tid] * is);
            atomicMax(&s_emax[par][ls_t], fx_exp(vt));
        }
        for (int j = tid + OC_THREADS; j < nv; j += OC_THREADS) {
            int ls = 0;
            while (s_sub0[ls + 1] <= v0 + j) ++ls;
            atomicMax(&s_emax[par][ls], fx_exp(fma(kdt, b_of(j, n + 1), yn[j] * is)));
        }
        if (b_t) b_next = b_t[(long long)min(n + 2, wp) * bK];
        __syncthreads();
        if (tid < nv) vl[tid] = fx_limbs(vt, s_emax[par][ls_t]);
        for (int j = tid + OC_THREADS; j < nv; j += OC_THREADS) {
            int ls = 0;
            while (s_sub0[ls + 1] <= v0 + j) ++ls;
            vl[j] = fx_limbs(fma(kdt, b_of(j, n + 1), yn[j] * is), s_emax[par][ls]);
        }
        if (tid >= OC_THREADS - OC_SUBS) s_emax[par ^ 1][tid - (OC_THREADS - OC_SUBS)] = 0;
        __syncthreads();
        const int i0 = (n % 3) * A.rows_max, i1 = ((n + 2) % 3) * A.rows_max, i2 = ((n + 1) % 3) * A.rows_max;
        // ---- own rows of y^{n+1} = G v and z^{n+1} = W v: 16 lanes a row, 8 on G, 8 on W
        const int half = (lane >> 3) & 1, l8 = lane & 7;
        double* ynext = yf + (par ^ 1) * A.nv_max;
        for (int base = 0; base < nr; base += 2 * OC_WARPS) {
            const int i = base + 2 * warp + (lane >> 4);
            long long s1 = 0, s2 = 0;
            int ls = 0, K = 0;
            if (i < nr) {
                ls = r_sub[i];
                K = s_sub0[ls + 1] - s_sub0[ls];
                const int2* g = lim + r_off[i] + half * oc_pitch(K);
                const int2* x = vl + (s_sub0[ls] - v0);
#pragma unroll 4
                for (int c = l8; c < K; c += 8) fx_mac2(s1, s2, g[c].x, g[c].y, x[c].x, x[c].y);
            }
            long long t = fx_fold(s1, s2);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) t += fx_shfl_xor(t, o);
            double y = 0.0;
            if (i < nr) {
                const int ev = s_emax[par][ls], eg = half ? r_ew[i] : r_eg[i];
                y = (double)t * fx_unit(ev, eg - 1022);
                if (ev == FX_BAD || eg >= FX_BAD) y = nan("");
            }
            const double z = __shfl_xor_sync(0xffffffffu, y, 8);
            if (i < nr) {
                const int r = r0 + i;
                if ((lane & 15) == 0) {
                    yo[i2 + i] = y;
                    zo[i2 + i] = z;
                    ps[i] = y * z;
                    v.arena[v.sub[in.sub_base + sA + ls].hist + (long long)(n + 1) * K + (r - s_sub0[ls])] = y;
                }
                // to the CTAs that hold rows of the same subdomain
                for (int p = lane & 15; p < CS; p += 16)
                    if (s_bound[p] < s_sub0[ls + 1] && s_bound[p + 1] > s_sub0[ls])
                        oc_store(ynext + (r - s_base[p]), (unsigned)p, half ? z : y);
            }
        }
        // ---- terms of D_n = || y^n/s_n - y^{n-1}/s_{n-1} ||^2
        for (int i = OC_THREADS - 1 - tid; i < nr; i += OC_THREADS)
            pd[i] = (n >= 1 && stop_rule)
                        ? (yo[i0 + i] * is - yo[i1 + i] * is_p) * (zo[i0 + i] * is - zo[i1 + i] * is_p)
                        : 0.0;
        __syncthreads();
        publish(par ^ 1);
        oc_sync();
    }
}

// ------------------------------------------------------------- host side

static cudaError_t oc_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int grid, int cs, size_t smem) {
    cudaError_t e = cudaFuncSetAttribute(k_window_onchip, cudaFuncAttributeMaxDynamicSharedMemorySize, OC_SMEM_MAX);
    if (e == cudaSuccess && cs > 8) e = cudaFuncSetAttribute(k_window_onchip, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg->gridDim = dim3((unsigned)grid);
    cfg->blockDim = dim3(OC_THREADS);
    cfg->dynamicSmemBytes = smem;
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return e;
}

// Rows of every instance dealt to clusters of `cs` CTAs by matrix elements.
// Returns false when a CTA's share does not fit its shared memory.
static bool oc_deal(const std::vector<InstDev>& inst, const std::vector<SubDev>& sub, int cs, OcPlan* p) {
    p->bounds.clear();
    p->row0.assign(sub.size(), 0);
    p->rows_max = p->nv_max = p->lim_max = 0;
    for (const InstDev& in : inst) {
        std::vector<int> cost, rsub;  // per row: limb pairs, subdomain
        for (int s = 0; s < in.n_sub; ++s) {
            const SubDev& sd = sub[in.sub_base + s];
            if (sd.K > OC_KMAX) return false;
            p->row0[in.sub_base + s] = (int)cost.size();
            if (cost.size() > 100000) return false;
            cost.insert(cost.end(), sd.K, 2 * oc_pitch(sd.K));
            rsub.insert(rsub.end(), sd.K, s);
        }
        long long total = 0, done = 0;
        for (int c : cost) total += c;
        size_t r = 0;
        for (int k = 0; k < cs; ++k) {
            const size_t first = r;
            p->bounds.push_back((int)first);
            long long lim = 0;
            while (r < cost.size() && (k == cs - 1 || done + cost[r] / 2 <= total * (k + 1) / cs)) {
                lim += cost[r];
                done += cost[r++];
            }
            // (an empty share keeps the subdomain of its first row)
            const int s0 = rsub[first < rsub.size() ? first : rsub.size() - 1], s1 = r > first ? rsub[r - 1] : s0;
            const int nv = p->row0[in.sub_base + s1] + sub[in.sub_base + s1].K - p->row0[in.sub_base + s0];
            if (s1 - s0 + 1 > OC_SUBS || lim > (1 << 20)) return false;
            if ((int)(r - first) > p->rows_max) p->rows_max = (int)(r - first);
            if (nv > p->nv_max) p->nv_max = nv;
            if (lim > p->lim_max) p->lim_max = (int)lim;
        }
        p->bounds.push_back((int)cost.size());
    }
    return oc_smem_bytes(p->rows_max, p->nv_max, p->lim_max) <= OC_SMEM_MAX;
}

// Launch shape of the on-chip window: the largest cluster of which the device
// holds one per instance at once and whose CTAs' shares fit; false when there
// is none (the two-phase window runs the problem).
bool oc_plan(const std::vector<InstDev>& inst, const std::vector<SubDev>& sub, int nsm, OcPlan* p) {
    const int ni = (int)inst.size();
    // about 24 rows per CTA (one pass of its warps) and more CTAs only for space:
    // 80 rows took 2.96 us a step on 4 CTAs, 3.25 on 16, 4.8 on one
    long long rows = 1;
    for (const InstDev& in : inst) {
        long long r = 0;
        for (int s = 0; s < in.n_sub; ++s) r += sub[in.sub_base + s].K;
        rows = r > rows ? r : rows;
    }
    int top = ni > 0 ? nsm / ni : 0;
    if (top > OC_CMAX) top = OC_CMAX;
    int start = (int)(rows < 24LL * top ? (rows + 23) / 24 : top);
    while (start >= 1 && start < top && !oc_deal(inst, sub, start, p)) ++start;
    for (int cs = start; cs >= 1; --cs) {
        if (!oc_deal(inst, sub, cs, p)) return false;  // fewer CTAs only take larger shares
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        int active = 0;
        if (oc_config(&cfg, at, ni * cs, cs, oc_smem_bytes(p->rows_max, p->nv_max, p->lim_max)) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&active, k_window_onchip, &cfg) == cudaSuccess && active >= ni) {
            p->cs = cs;
            return true;
        }
        cudaGetLastError();
    }
    return false;
}

cudaError_t launch_oc_make_w(const SwrDeviceView& v, cudaStream_t st, int max_K) {
    k_oc_make_w<<<dim3((unsigned)max_K, v.n_sub), 128, 0, st>>>(v);
    return cudaGetLastError();
}

cudaError_t launch_oc_window(const SweepArgs& s, const OcPlan& p, const int* d_bounds, const int* d_row0, cudaStream_t st) {
    OcArgs a;
    a.v = s.v;
    a.bounds = d_bounds;
    a.row0 = d_row0;
    a.win_prev = s.win_prev;
    a.snorm = s.snorm;
    a.win = s.win;
    a.n_active = s.n_active;
    a.cap = s.cap;
    a.cs = p.cs;
    a.tune_steps = s.tune_steps;
    a.rows_max = p.rows_max;
    a.nv_max = p.nv_max;
    a.lim_max = p.lim_max;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cudaError_t e = oc_config(&cfg, at, s.v.n_inst * p.cs, p.cs, oc_smem_bytes(p.rows_max, p.nv_max, p.lim_max));
    if (e != cudaSuccess) return e;
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, k_window_onchip, a);
}

}  // namespace swr
