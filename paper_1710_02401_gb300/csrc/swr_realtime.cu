// swr_realtime.cu -- the real-time window (Crank-Nicolson under the dipole
// field) as one persistent kernel.
//
// The step is the one stated in swr_tdse.cu:
//   r = 2 c^n + i (theta_{n+1} - theta_n) Q' c^n + i dt/2 kappa (b'^{n+1} + b'^n),
//   (M0 + i theta_{n+1} Q') x = r,   c^{n+1} = x - c^n,
// by the fixed point x <- G0 (r - i theta_{n+1} Q' x), G0 = M0^{-1}, which
// contracts with rho = |theta_{n+1}| max_{Omega_i} |x_1 + ... + x_N| (||G0|| <= 1).
// Within a Schwarz iteration the subdomains' windows do not depend on one
// another, so one cluster of CTAs carries one subdomain through all its steps;
// nothing waits for another subdomain and the host launches one kernel
// (before: three launches per sweep, a thousand-node graph per iteration kind).
//
// Three things set the time:
//  - G0 is complex symmetric (H' real symmetric, R' symmetric): only its lower
//    triangle is read, each element used for its row and its column.  At
//    K = 1024 a sweep streams 8 bytes per element of the full matrix from HBM
//    instead of 16.  Smaller matrices stay in shared memory for the window.
//  - The products run in 56-bit fixed point on the integer pipes
//    (swr_fixed.cuh), complex ones as three real products (Karatsuba; sums are
//    exact, so nothing cancels): 6 real multiply-adds per clock and SM against
//    1.6 on the FP64 pipe, which was 94 % busy on the FP64 path, and more exact
//    than the double-single sums of the mixed path at the same instruction
//    count.  Both precisions run this kernel.  It is bound by the integer
//    multiplier: at K = 1024 with 64 subdomains (2 CTAs each) a sweep takes
//    190 us, 2.8 TB/s of the halved matrix; 8 warps of 240 registers with
//    4 x 4 elements per lane measured the same as 16 of 128 (203 us).
//  - The fixed point starts from the sixth-order extrapolation x_g of
//    c^{n+1} + c^n and iterates on d = x - x_g,
//      u_0 = 2 c^n + i hk B + i Q' [(theta_{n+1} - theta_n) c^n - theta_{n+1} x_g],
//      x_m = G0 u_{m-1},  u_m = u_0 - i theta_{n+1} Q' d_m,
//    until rho / (1 - rho) ||x_m - x_{m-1}|| <= 1e-15 ||x_m||: the same bound on
//    what is left as the a-priori count from x = 0 gave (rho^(m+1) <= 1e-15),
//    reached in 4.6 instead of 7.2 sweeps on the 16-subdomain learned-trace
//    problems (6.1 with one point); where the fine basis carries unresolved
//    frequencies (K = 1024) it gains nothing (3.7).
// Window of one Schwarz iteration, before and now: 64 subdomains of K = 1024,
// 250 steps, mixed 233 -> 178 ms, FP64 (100 steps) 177 -> 60 ms; 192 of K = 100,
// 100 steps, FP64 68 -> 10.7 ms.
//
// Layout of G0: in place of the inverse (16 bytes per element, row-major) the
// limbs (re hi, re lo, im hi, im lo), each strip of 8 rows rearranged inside its
// own space into chunks of 64 columns, [chunk][row][column], the lower triangle
// only (the last chunk of a strip ends with the strip's last diagonal
// element): a chunk is one contiguous bulk copy.  A sweep walks 64 x 64 tiles of
// the lower triangle, block column by block column, the cluster's CTAs taking
// equal runs of tiles; warp w of a CTA streams strip w of each tile through its
// own ring of bulk copies (no CTA barrier inside a sweep).  Lanes own 4 rows x 4
// columns each: row sums are reduced over 16 lanes per tile, column sums stay
// in registers over a block column.  Integer sums are exact, so partial results
// may be added in any order.
//
// Every wait of a bulk copy is bounded: spin_limit / 16 polls, since a poll
// suspends for about 16 polls of an ordinary flag.  A warp that gives up raises
// SWR_ERR_TIMEOUT, reads no further stage and issues no further copy, and its CTA
// tells the cluster through the norm exchange, after which all leave together,
// each once its own copies in flight have landed (a wait that does not follow the
// caller's limit: a CTA must not exit while a copy still writes its shared
// memory, and a copy of 8 KB completes within microseconds).
#include <math.h>

#include "swr_fixed.cuh"

namespace swr {

#define RT_THREADS 256
#define RT_WARPS (RT_THREADS / 32)
#define RT_T 64                              // tile edge
#define RT_S (RT_T / RT_WARPS)               // rows of a strip (a warp's share of a tile)
#define RT_LR (RT_S / 2)                      // rows of a lane
#define RT_CHUNK (RT_S * RT_T * 16)          // bytes of a strip's columns of a tile
#define RT_NST_MAX 8
#define RT_EXTRAP 6                          // points of the extrapolation
#define RT_SWEEPS_MAX 64
#define RT_SMEM_MAX (225 * 1024)

__device__ inline unsigned rt_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ inline unsigned rt_map(const void* local, unsigned rank) {
    unsigned ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(rt_smem(local)), "r"(rank));
    return ra;
}
__device__ inline void rt_store2(const void* local, unsigned rank, double a, double b) {
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(rt_map(local, rank)), "d"(a), "d"(b) : "memory");
}
__device__ inline void rt_store2f(const void* local, unsigned rank, float a, float b) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(rt_map(local, rank)), "f"(a), "f"(b) : "memory");
}
__device__ inline longlong2 rt_load2(const void* local, unsigned rank) {
    longlong2 v;
    asm volatile("ld.shared::cluster.v2.s64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(rt_map(local, rank)) : "memory");
    return v;
}
__device__ inline void rt_sync(int cs) {
    if (cs > 1) asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    else __syncthreads();
}
__device__ inline bool rt_wait(unsigned mbar, unsigned parity, long long limit) {
    for (long long it = 0; it < limit; ++it) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// (-1)^j C(np, j + 1): weights of c^{n-j} in the extrapolation from np points.
__constant__ double RT_W[RT_EXTRAP][RT_EXTRAP] = {{1, 0, 0, 0, 0, 0},     {2, -1, 0, 0, 0, 0},      {3, -3, 1, 0, 0, 0},
                                                  {4, -6, 4, -1, 0, 0},   {5, -10, 10, -5, 1, 0},   {6, -15, 20, -15, 6, -1}};

struct RtArgs {
    SwrDeviceView v;
    const long long* boff;    // per subdomain three vectors of 2 K doubles (u_0, x_g, d)
    const int* win_prev;
    const double* theta;      // [n_inst][cap + 1] dt/2 e(t_n)
    unsigned* sweeps;         // [n_sub] matrix sweeps of the window
    const int* gexp;          // [n_sub] exponent of G0 (k_rt_scale)
    long long spin_limit;
    int cap, cs, kmax, qel, nst, own_smem;  // qel: elements of the Q' factors (both coordinates)
};

// theta_n = dt/2 e(t_n), n = 0 .. cap, per instance (the FP64 sines take
// microseconds on one thread: once per window here, not in every step).
__global__ void k_rt_theta(SwrDeviceView v, double* theta, int cap) {
    const InstDev& in = v.inst[blockIdx.y];
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n > cap) return;
    const double t = n * in.dt;
    double e = 0.0;
    if (in.E0 != 0.0 && t >= 0.0 && t <= in.T) {
        const double s = sin(M_PI * t / in.T);
        e = in.E0 * s * s * sin(in.omega * t + in.phase);
    }
    theta[(long long)blockIdx.y * (cap + 1) + n] = 0.5 * in.dt * e;
}

// Exponent of a subdomain's G0, the largest of its rows' (fx_row_exp: 2^0 for the ||G0|| <= 1 of an
// absorbing boundary with kinetic > 0; larger where G0 is, smaller where the
// whole matrix is small), FX_BAD when an entry is not finite.  A warp per row.
__global__ void k_rt_scale(SwrDeviceView v, int* gexp) {
    const SubDev& s = v.sub[blockIdx.y];
    const int K = s.K, lane = threadIdx.x & 31, r = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (r >= K) return;
    const double2* g = reinterpret_cast<const double2*>(v.arena + s.Gm) + (size_t)r * K;
    int e = 0;
    for (int c = lane; c < K; c += 32) e = max(e, max(fx_exp(g[c].x), fx_exp(g[c].y)));
    e = __reduce_max_sync(0xffffffffu, e);
    const double sc = fx_row_scale(e);
    float q = 0.f;
    for (int c = lane; c < K; c += 32) {
        const float a = (float)(g[c].x * sc), b = (float)(g[c].y * sc);
        q += a * a + b * b;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if (lane == 0) atomicMax(gexp + blockIdx.y, fx_row_exp(e, q));
}

// Limbs of the lower triangle of G0 relative to its exponent, strip by strip
// in place through shared memory: columns of the chunk of block column J have
// the pitch min(64, columns up to the strip's last row).
__global__ void k_rt_pack(SwrDeviceView v, const int* gexp) {
    extern __shared__ int4 rt_strip[];
    const SubDev& s = v.sub[blockIdx.y];
    const int K = s.K, r0 = blockIdx.x * RT_S, eg = gexp[blockIdx.y];
    if (r0 >= K) return;
    const int nr = min(RT_S, K - r0), nc = min(K, r0 + RT_S);  // columns kept of every row of the strip
    double2* G = reinterpret_cast<double2*>(v.arena + s.Gm) + (size_t)r0 * K;
    for (int e = threadIdx.x; e < nr * nc; e += blockDim.x) {
        const int i = e / nc, c = e - i * nc, J = c / RT_T, pitch = min(RT_T, nc - J * RT_T);
        const double2 g = G[(size_t)i * K + c];
        const int2 a = fx_limbs(g.x, eg), b = fx_limbs(g.y, eg);
        rt_strip[J * nr * RT_T + i * pitch + c - J * RT_T] = make_int4(a.x, a.y, b.x, b.y);
    }
    __syncthreads();
    // (all of the strip is read; its nr x nc elements, the chunks one after another)
    for (int e = threadIdx.x; e < nr * nc; e += blockDim.x) reinterpret_cast<int4*>(G)[e] = rt_strip[e];
}

// Largest exponent field of n (value, value) pairs, over the CTA; FX_BAD when a
// value is not finite.
__device__ inline int rt_max_exp(const double2* x, int n, int* s_max) {
    int e = 0;
    for (int i = threadIdx.x; i < n; i += RT_THREADS) e = max(e, max(fx_exp(x[i].x), fx_exp(x[i].y)));
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = e;
    __syncthreads();
    e = s_max[0];
#pragma unroll
    for (int w = 1; w < RT_WARPS; ++w) e = max(e, s_max[w]);
    return e;
}
// FP64 pairs -> limbs in place; returns the exponent.
__device__ inline int rt_to_limbs(double2* x, int n, int* s_max) {
    const int e = rt_max_exp(x, n, s_max);
    for (int i = threadIdx.x; i < n; i += RT_THREADS) {
        const double2 q = x[i];
        const int2 a = fx_limbs(q.x, e), b = fx_limbs(q.y, e);
        reinterpret_cast<int4*>(x)[i] = make_int4(a.x, a.y, b.x, b.y);
    }
    __syncthreads();  // also: s_max may be written again
    return e;
}

// Position in the CTA's run of tiles [t0, t1) of the lower triangle, block column
// by block column; tiles in which this warp has no rows are passed over.
struct RtCursor {
    int J, I, id;
    __device__ inline void next(int T, int t0, int t1, int J0, int I0, int last_skip) {
        do {
            if (++id == t1) {
                id = t0;
                J = J0;
                I = I0;
            } else if (++I == T) {
                ++J;
                I = J;
            }
        } while (last_skip && I == T - 1);
    }
};

// A complex operand (c + i d) as limbs of c, d - c and c + d (hi, lo each).
struct RtOp {
    int ch, cl, mh, ml, ph, pl;
};
__device__ inline RtOp rt_op(int4 u) { return {u.x, u.y, u.z - u.x, u.w - u.y, u.x + u.z, u.y + u.w}; }

// One warp's strip of a tile, lanes RT_LR rows x 4 columns: row sums to rv (re,
// im per row, folded), column sums added to cs (three partial products per
// column).  (a + i b)(c + i d) = k1 - k3 + i (k1 + k2), k1 = (a + b) c,
// k2 = a (d - c), k3 = b (c + d).  Row and column use every element of the
// chunk once each.  DIAG: rr0 = the lane's first row, c0 = its first column in
// the tile; elements above the diagonal are not there, the diagonal counts once.
template <bool DIAG>
__device__ inline void rt_tile(const int4* g, int pitch, const int4* uI, const RtOp (&vj)[4], long long (&cs)[12],
                               long long (&rv)[2 * RT_LR], int rr0, int c0) {
    long long c2[12];
#pragma unroll
    for (int j = 0; j < 12; ++j) c2[j] = 0;
#pragma unroll
    for (int i = 0; i < RT_LR; ++i) {
        const RtOp u = rt_op(uI[i]);
        long long k1 = 0, k2 = 0, k3 = 0, l1 = 0, l2 = 0, l3 = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int4 e = g[i * pitch + 16 * j], f;
            f = e;
            if (DIAG) {
                const int d = c0 + 16 * j - (rr0 + i);
                if (d > 0) e = make_int4(0, 0, 0, 0);
                if (d >= 0) f = make_int4(0, 0, 0, 0);
            }
            const int sh = e.x + e.z, sl = e.y + e.w, th = DIAG ? f.x + f.z : sh, tl = DIAG ? f.y + f.w : sl;
            fx_mac2(k1, l1, sh, sl, vj[j].ch, vj[j].cl);
            fx_mac2(cs[3 * j], c2[3 * j], th, tl, u.ch, u.cl);
            fx_mac2(k2, l2, e.x, e.y, vj[j].mh, vj[j].ml);
            fx_mac2(cs[3 * j + 1], c2[3 * j + 1], f.x, f.y, u.mh, u.ml);
            fx_mac2(k3, l3, e.z, e.w, vj[j].ph, vj[j].pl);
            fx_mac2(cs[3 * j + 2], c2[3 * j + 2], f.z, f.w, u.ph, u.pl);
        }
        rv[2 * i] = fx_fold(k1 - k3, l1 - l3);
        rv[2 * i + 1] = fx_fold(k1 + k2, l1 + l2);
    }
#pragma unroll
    for (int j = 0; j < 12; ++j) cs[j] = fx_fold(cs[j], c2[j]);
}

__global__ void __launch_bounds__(RT_THREADS, 1) k_rt_window(RtArgs A) {
    extern __shared__ __align__(128) unsigned char rt_sm[];
    __shared__ __align__(8) unsigned long long s_bar[RT_WARPS][RT_NST_MAX];
    __shared__ int s_max[RT_WARPS];
    __shared__ float2 s_red[RT_WARPS];
    __shared__ __align__(8) float2 s_norm[16];  // per CTA of the cluster: ||x_m - x_{m-1}||^2, ||x_m||^2 (< 0: gave up)
    __shared__ int s_fail;
    const SwrDeviceView& v = A.v;
    const int CS = A.cs, sid = blockIdx.x / CS;
    const unsigned rank = blockIdx.x % CS;
    const SubDev& s = v.sub[sid];
    const InstDev& in = v.inst[s.inst];
    if (in.anti && s.N == 2 && s.idx[0] > s.idx[1]) return;  // mirror image of another subdomain (whole cluster)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lr = lane >> 4, lc = lane & 15;
    const int K = s.K, kd = s.kd, T = (K + RT_T - 1) / RT_T, Kp = T * RT_T;
    const int Km = (A.kmax + RT_T - 1) / RT_T * RT_T, nst = A.nst;
    unsigned char* ring = rt_sm + (size_t)warp * nst * RT_CHUNK;
    double2* ul = reinterpret_cast<double2*>(rt_sm + (size_t)RT_WARPS * nst * RT_CHUNK);  // u, then its limbs
    longlong2* yr = reinterpret_cast<longlong2*>(ul + Km);                                // row sums
    longlong2* yc = yr + Km;                                                              // column sums
    double2* xs = reinterpret_cast<double2*>(yc + Km);                                    // argument of Q', then its limbs
    int2* X1t = reinterpret_cast<int2*>(xs + Km);                                         // [c][a]
    int2* X2 = X1t + kd * kd;
    const int ra = (int)((long long)K * rank / CS), rb = (int)((long long)K * (rank + 1) / CS);  // own rows
    double2 *u0, *xg, *dp;  // own rows: u_0, x_g, d of the sweep before (index r - ra)
    if (A.own_smem) {
        const int rm = (A.kmax + CS - 1) / CS;
        u0 = reinterpret_cast<double2*>(X1t + A.qel);
        xg = u0 + rm;
        dp = xg + rm;
    } else {
        u0 = reinterpret_cast<double2*>(v.arena + A.boff[3 * sid]) + ra;
        xg = reinterpret_cast<double2*>(v.arena + A.boff[3 * sid + 1]) + ra;
        dp = reinterpret_cast<double2*>(v.arena + A.boff[3 * sid + 2]) + ra;
    }
    const unsigned char* G = reinterpret_cast<const unsigned char*>(v.arena + s.Gm);
    const long long limit = A.spin_limit >> 4;
    const long long copy_limit = limit > (1LL << 20) ? limit : (1LL << 20);

    // ------------------------------------------------------------ the ring
    const int nt = T * (T + 1) / 2, t0 = (int)((long long)nt * rank / CS), t1 = (int)((long long)nt * (rank + 1) / CS);
    const int last_skip = (T - 1) * RT_T + warp * RT_S >= K;  // this warp has no rows in the last block row
    int J0 = 0, I0 = 0;
    for (int id = 0; id < t0; ++id)
        if (++I0 == T) {
            ++J0;
            I0 = J0;
        }
    int nact = 0;  // this warp's tiles of a sweep
    {
        int J = J0, I = I0;
        for (int id = t0; id < t1; ++id) {
            if (!(last_skip && I == T - 1)) ++nact;
            if (++I == T) {
                ++J;
                I = J;
            }
        }
    }
    const bool resident = nact <= nst;
    RtCursor ld{J0, I0, t0}, cp{J0, I0, t0};
    if (nact > 0 && last_skip && I0 == T - 1) {
        ld.next(T, t0, t1, J0, I0, last_skip);
        cp = ld;
    }
    unsigned qload = 0, qcomp = 0;
    // strip w of the tile under the load cursor into the next stage
    auto issue = [&]() {
        const unsigned st = qload % nst, bar = rt_smem(&s_bar[warp][st]);
        const int r0 = ld.I * RT_T + warp * RT_S, nr = min(RT_S, K - r0);
        const int pitch = min(RT_T, min(K, r0 + RT_S) - ld.J * RT_T);
        const unsigned bytes = (unsigned)(nr * pitch * 16);
        if (lane == 0) {
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                             rt_smem(ring + (size_t)st * RT_CHUNK)),
                         "l"(G + ((size_t)r0 * K + ld.J * nr * RT_T) * 16), "r"(bytes), "r"(bar)
                         : "memory");
        }
        ++qload;
        ld.next(T, t0, t1, J0, I0, last_skip);
    };

    // ------------------------------------------------------------- set-up
    if (lane == 0) {
        for (int i = 0; i < nst; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(rt_smem(&s_bar[warp][i])));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid == 0) s_fail = 0;
    __syncwarp();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    for (int i = 0; i < min(nst, nact); ++i) issue();
    for (int i = tid; i < Kp; i += RT_THREADS) {
        ul[i] = xs[i] = make_double2(0.0, 0.0);
        yr[i] = yc[i] = make_longlong2(0, 0);
    }
    // Q' factors as limbs with a common exponent (the first transposed: a warp's
    // consecutive rows read consecutive words)
    int eX;
    {
        T1Layout lay(s.q, kd);
        const double* X1g = v.arena + s.t1[0] + lay.mat(M_XP);
        const double* X2g = v.arena + s.t1[s.N == 2 ? 1 : 0] + lay.mat(M_XP);
        int e = 0;
        for (int i = tid; i < kd * kd; i += RT_THREADS) e = max(e, max(fx_exp(X1g[i]), fx_exp(X2g[i])));
        e = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0) s_max[warp] = e;
        __syncthreads();
        eX = s_max[0];
        for (int w = 1; w < RT_WARPS; ++w) eX = max(eX, s_max[w]);
        for (int i = tid; i < kd * kd; i += RT_THREADS) {
            const int a = i / kd, c = i - a * kd;
            X1t[c * kd + a] = fx_limbs(X1g[i], eX);
            if (s.N == 2) X2[i] = fx_limbs(X2g[i], eX);
        }
    }
    const int wp = A.win_prev[s.inst];
    const double* hist = v.arena + s.hist;
    const double* bvec = v.arena + s.bvec;
    const double* theta = A.theta + (long long)s.inst * (A.cap + 1);
    const double hk = 0.5 * in.dt * in.kappa;
    const int eg = A.gexp[sid] - 1022;  // G0 = limbs x 2^(eg - 56)
    double qlo = 0, qhi = 0;
    for (int e = 0; e < s.N; ++e) {
        qlo += s.lo[e];
        qhi += s.hi[e];
    }
    const float qn = (float)fmax(fabs(qlo), fabs(qhi));
    const int nsteps = in.window_cap;
    unsigned nsweeps = 0;
    for (int r = ra + tid; r < rb; r += RT_THREADS) {
        double* h0 = v.arena + s.hist;
        h0[r] = v.arena[s.c0 + r];
        h0[K + r] = v.arena[s.c0 + K + r];
    }
    rt_sync(CS);  // every CTA initialised before the first remote store

    // Q' z for own rows, z the limbs in xs (exponent ez): calls f(r, re, im)
    auto apply_q = [&](int ez, auto f) {
        const double unit = fx_unit(ez, eX - 1022);
        const double bad = (ez == FX_BAD || eX == FX_BAD) ? nan("") : 0.0;
        const int4* z = reinterpret_cast<const int4*>(xs);
        for (int r = ra + tid; r < rb; r += RT_THREADS) {
            long long r1 = 0, r2 = 0, i1 = 0, i2 = 0;
            if (s.N == 1) {
                for (int c = 0; c < kd; ++c) {
                    const int2 x = X1t[c * kd + r];
                    const int4 q = z[c];
                    fx_mac2(r1, r2, x.x, x.y, q.x, q.y);
                    fx_mac2(i1, i2, x.x, x.y, q.z, q.w);
                }
            } else {
                const int b = r / kd, a = r - b * kd;
#pragma unroll 4
                for (int c = 0; c < kd; ++c) {
                    const int2 x = X1t[c * kd + a];
                    const int4 q = z[c + kd * b];
                    fx_mac2(r1, r2, x.x, x.y, q.x, q.y);
                    fx_mac2(i1, i2, x.x, x.y, q.z, q.w);
                }
#pragma unroll 4
                for (int e = 0; e < kd; ++e) {
                    const int2 x = X2[b * kd + e];
                    const int4 q = z[a + kd * e];
                    fx_mac2(r1, r2, x.x, x.y, q.x, q.y);
                    fx_mac2(i1, i2, x.x, x.y, q.z, q.w);
                }
            }
            f(r, (double)fx_fold(r1, r2) * unit + bad, (double)fx_fold(i1, i2) * unit + bad);
        }
    };

    // this warp's share of y = G0 u (limbs in ul) into yr, yc
    auto sweep = [&]() {
        const int4* U = reinterpret_cast<const int4*>(ul);
        RtOp vj[4];
        long long cs[12];
        int J = -1;
        auto flush = [&]() {
            const bool up = lane & 16;  // lanes of row group 0 end with columns 0, 1, of group 1 with 2, 3
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int col = J * RT_T + lc + 16 * ((up ? 2 : 0) + j);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const long long a = h ? cs[3 * j] + cs[3 * j + 1] : cs[3 * j] - cs[3 * j + 2];
                    const long long b = h ? cs[3 * j + 6] + cs[3 * j + 7] : cs[3 * j + 6] - cs[3 * j + 8];
                    const long long val = (up ? b : a) + fx_shfl_xor(up ? a : b, 16);
                    atomicAdd(reinterpret_cast<unsigned long long*>(yc) + 2 * col + h, (unsigned long long)val);
                }
            }
        };
        for (int t = 0; t < nact; ++t) {
            const unsigned st = resident ? (unsigned)t : qcomp % nst, par = resident ? 0u : (qcomp / nst) & 1u;
            if (cp.J != J) {
                if (J >= 0) flush();
                J = cp.J;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    vj[j] = rt_op(U[J * RT_T + lc + 16 * j]);
                    cs[3 * j] = cs[3 * j + 1] = cs[3 * j + 2] = 0;
                }
            }
            if (!__all_sync(0xffffffffu, rt_wait(rt_smem(&s_bar[warp][st]), par, limit))) {
                s_fail = 1;
                if (lane == 0) atomicOr(v.err, SWR_ERR_TIMEOUT);
                break;
            }
            const int4* g = reinterpret_cast<const int4*>(ring + (size_t)st * RT_CHUNK) + lc;
            const int rr0 = warp * RT_S + lr * RT_LR;
            const int4* uI = U + cp.I * RT_T + rr0;
            long long rv[2 * RT_LR];
            if (cp.I == cp.J) {
                const int pitch = min(RT_T, min(K - cp.J * RT_T, (warp + 1) * RT_S));
                rt_tile<true>(g + lr * RT_LR * pitch, pitch, uI, vj, cs, rv, rr0, lc);
            } else {
                rt_tile<false>(g + lr * RT_LR * RT_T, RT_T, uI, vj, cs, rv, rr0, lc);
            }
            // the stage is read: refill it
            __syncwarp();
            if (!resident) {
                ++qcomp;
                issue();
            }
            // row sums over the 16 lanes of a row group: the upper lane bits end up choosing the value
#pragma unroll
            for (int o = 8, n = 2 * RT_LR; o >= 1; o >>= 1, n >>= 1) {
                const bool up = lane & o;
                if (n > 1) {
#pragma unroll
                    for (int j = 0; j < RT_LR; ++j)
                        if (j < n / 2) {
                            const long long send = up ? rv[j] : rv[j + n / 2], keep = up ? rv[j + n / 2] : rv[j];
                            rv[j] = keep + fx_shfl_xor(send, o);
                        }
                } else {
                    rv[0] += fx_shfl_xor(rv[0], o);
                }
            }
            if (!(lane & (8 / RT_LR - 1))) {
                const int idx = lc / (8 / RT_LR);
                long long* y = reinterpret_cast<long long*>(yr) + 2 * (cp.I * RT_T + rr0 + (idx >> 1)) + (idx & 1);
                *y += rv[0];
            }
            cp.next(T, t0, t1, J0, I0, last_skip);
        }
        if (J >= 0) flush();
    };

    bool failed = false;
    for (int n = 0; n < nsteps && !failed; ++n) {
        // ---- own rows: c^n, the extrapolated x_g, z = (theta_{n+1} - theta_n) c^n - theta_{n+1} x_g
        const double th1 = theta[n + 1], dth = th1 - theta[n];
        const double* b1 = wp > 0 ? bvec + (long long)min(n + 1, wp) * 2 * K : nullptr;
        const double* b0 = wp > 0 ? bvec + (long long)min(n, wp) * 2 * K : nullptr;
        const int np = min(RT_EXTRAP, n + 1);
        for (int r = ra + tid; r < rb; r += RT_THREADS) {
            // c^{n+1} ~ sum_j (-1)^j C(np, j + 1) c^{n-j}
            double cr[RT_EXTRAP], ci[RT_EXTRAP];
#pragma unroll
            for (int j = 0; j < RT_EXTRAP; ++j) {
                cr[j] = j < np ? hist[(long long)(n - j) * 2 * K + r] : 0.0;
                ci[j] = j < np ? hist[(long long)(n - j) * 2 * K + K + r] : 0.0;
            }
            double gr = cr[0], gi = ci[0];
#pragma unroll
            for (int j = 0; j < RT_EXTRAP; ++j) {
                gr = fma(RT_W[np - 1][j], cr[j], gr);
                gi = fma(RT_W[np - 1][j], ci[j], gi);
            }
            xg[r - ra] = make_double2(gr, gi);
            dp[r - ra] = make_double2(0.0, 0.0);
            const double zr = dth * cr[0] - th1 * gr, zi = dth * ci[0] - th1 * gi;
            double br = 0.0, bi = 0.0;
            if (b1) {
                br = b1[r] + b0[r];
                bi = b1[K + r] + b0[K + r];
            }
            u0[r - ra] = make_double2(2.0 * cr[0] - hk * bi, 2.0 * ci[0] + hk * br);
            for (int p = 0; p < CS; ++p) rt_store2(xs + r, p, zr, zi);
        }
        for (int i = tid; i < Kp; i += RT_THREADS) yr[i] = yc[i] = make_longlong2(0, 0);
        rt_sync(CS);
        int ez = rt_to_limbs(xs, Kp, s_max);
        apply_q(ez, [&](int r, double qr, double qi) {
            const double2 b = u0[r - ra];
            const double a = b.x - qi, c = b.y + qr;  // + i Q' z
            u0[r - ra] = make_double2(a, c);
            for (int p = 0; p < CS; ++p) rt_store2(ul + r, p, a, c);
        });
        const float rho = fabsf((float)th1) * qn;
        const float rfac = rho / (1.0f - rho);
        for (int m = 1;; ++m) {
            rt_sync(CS);
            const int eu = rt_to_limbs(ul, Kp, s_max);
            sweep();
            ++nsweeps;
            rt_sync(CS);
            // ---- own rows of x_m, d_m = x_m - x_g and the norms of the stop test
            const double unit = fx_unit(eu, eg), bad = eu == FX_BAD || eg >= FX_BAD - 1022 ? nan("") : 0.0;
            const int en = 2045 - eu - eg;  // scales the norms to units of 2^56 sums
            const double inv = en > 0 && en < 0x7ff ? __hiloint2double(en << 20, 0) : 0.0;
            float nd = 0.f, nx = 0.f;
            for (int r = ra + tid; r < rb; r += RT_THREADS) {
                long long sr = 0, si = 0;
                for (int p = 0; p < CS; ++p) {
                    const longlong2 a = rt_load2(yr + r, p), c = rt_load2(yc + r, p);
                    sr += a.x + c.x;
                    si += a.y + c.y;
                }
                const double2 g = xg[r - ra], d0 = dp[r - ra];
                const double dr = ((double)sr * unit + bad) - g.x, di = ((double)si * unit + bad) - g.y;
                dp[r - ra] = make_double2(dr, di);
                const float er = (float)((dr - d0.x) * inv), ei = (float)((di - d0.y) * inv);
                const float fr = (float)sr * 1.3877788e-17f, fi = (float)si * 1.3877788e-17f;  // 2^-56
                nd += er * er + ei * ei;
                nx += fr * fr + fi * fi;
                for (int p = 0; p < CS; ++p) rt_store2(xs + r, p, dr, di);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                nd += __shfl_xor_sync(0xffffffffu, nd, o);
                nx += __shfl_xor_sync(0xffffffffu, nx, o);
            }
            if (lane == 0) s_red[warp] = make_float2(nd, nx);
            __syncthreads();
            if (tid < CS) {
                float a = 0.f, b = 0.f;
                for (int w = 0; w < RT_WARPS; ++w) {
                    a += s_red[w].x;
                    b += s_red[w].y;
                }
                rt_store2f(&s_norm[rank], tid, a, s_fail ? -1.0f : b);
            }
            rt_sync(CS);
            nd = nx = 0.f;
            for (int p = 0; p < CS; ++p) {
                const float2 q = s_norm[p];
                nd += q.x;
                nx += q.y;
                failed = failed || q.y < 0.f;
            }
            // converged (also when a value is not finite: the residual reports it)
            if (failed || !(rfac * sqrtf(nd) > 1e-15f * sqrtf(nx)) || m >= RT_SWEEPS_MAX) break;
            for (int i = tid; i < Kp; i += RT_THREADS) yr[i] = yc[i] = make_longlong2(0, 0);
            ez = rt_to_limbs(xs, Kp, s_max);
            apply_q(ez, [&](int r, double qr, double qi) {
                const double2 b = u0[r - ra];
                const double a = b.x + th1 * qi, c = b.y - th1 * qr;  // - i theta Q' d
                for (int p = 0; p < CS; ++p) rt_store2(ul + r, p, a, c);
            });
        }
        // ---- c^{n+1} = x - c^n, x = x_g + d
        double* hn = v.arena + s.hist + (long long)(n + 1) * 2 * K;
        for (int r = ra + tid; r < rb; r += RT_THREADS) {
            const double2 g = xg[r - ra], d = dp[r - ra];
            hn[r] = (g.x + d.x) - hist[(long long)n * 2 * K + r];
            hn[K + r] = (g.y + d.y) - hist[(long long)n * 2 * K + K + r];
        }
    }
    // copies in flight (the next sweep's first chunks) before the CTA leaves
    for (unsigned q = resident ? 0u : qcomp; q < qload; ++q) rt_wait(rt_smem(&s_bar[warp][q % nst]), (q / nst) & 1u, copy_limit);
    if (rank == 0 && tid == 0) A.sweeps[sid] = nsweeps;
}

// ------------------------------------------------------------- host side

static size_t rt_smem_bytes(int kmax, int qel, int cs, int nst, bool own) {
    const size_t km = (size_t)(kmax + RT_T - 1) / RT_T * RT_T;
    return (size_t)RT_WARPS * nst * RT_CHUNK + 4 * km * 16 + (((size_t)qel + 1) & ~(size_t)1) * sizeof(int2) +
           (own ? 3 * (size_t)((kmax + cs - 1) / cs) * 16 : 0);
}

static cudaError_t rt_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int n_sub, int cs, size_t smem) {
    cudaError_t e = cudaFuncSetAttribute(k_rt_window, cudaFuncAttributeMaxDynamicSharedMemorySize, RT_SMEM_MAX);
    if (e == cudaSuccess && cs > 8) e = cudaFuncSetAttribute(k_rt_window, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg->gridDim = dim3((unsigned)(n_sub * cs));
    cfg->blockDim = dim3(RT_THREADS);
    cfg->dynamicSmemBytes = smem;
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return e;
}

// Launch shape of the window: CTAs per subdomain, ring stages per warp and
// whether the own-row vectors fit shared memory.  Per cluster size the ring
// takes as many stages as hold a CTA's tiles (the matrix then stays on chip) or
// fit; the size is the one with the least waves x (tiles per CTA + overhead of a
// sweep in tile times: about half for one CTA, 2.5 with cluster barriers).
// A subdomain gets 16 CTAs at most, also when it is alone on the chip: 70 us a step
// at K = 1024, where sweeps over the whole chip launched one by one took 162 (FP64)
// and 103 (double-single).  Returns false when no shape fits.
bool rt_plan(int n_sub, int kmax, int qel, RtPlan* out) {
    const int T = (kmax + RT_T - 1) / RT_T, nt = T * (T + 1) / 2;
    double best = 1e300;
    for (int c = 1; c <= 16 && (c == 1 || 2 * c <= nt); ++c) {
        const int want = (nt + c - 1) / c;
        int nst = 0;
        bool own = true;
        for (int pass = 0; pass < 2 && nst == 0; ++pass) {
            own = pass == 0;
            for (int n = want < RT_NST_MAX ? want : RT_NST_MAX; n >= (own && want > 1 ? 2 : 1) && nst == 0; --n)
                if (rt_smem_bytes(kmax, qel, c, n, own) <= RT_SMEM_MAX) nst = n;
        }
        if (nst == 0) continue;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        int active = 0;
        if (rt_config(&cfg, at, n_sub, c, rt_smem_bytes(kmax, qel, c, nst, own)) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&active, k_rt_window, &cfg) != cudaSuccess || active < 1) {
            cudaGetLastError();
            continue;
        }
        const double cost = (double)((n_sub + active - 1) / active) * (want + (c > 1 ? 2.5 : 0.5));
        if (cost < best) {
            best = cost;
            out->cs = c;
            out->nst = nst;
            out->own = own ? 1 : 0;
        }
    }
    return best < 1e300;
}

cudaError_t launch_rt_pack(const SwrDeviceView& v, cudaStream_t st, int max_K, int* d_gexp) {
    const int T = (max_K + RT_T - 1) / RT_T;
    const size_t smem = (size_t)T * RT_S * RT_T * sizeof(int4);
    cudaError_t e = allow_dynamic_smem((const void*)k_rt_pack);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_gexp, 0, v.n_sub * sizeof(int), st);
    if (e != cudaSuccess) return e;
    k_rt_scale<<<dim3((unsigned)((max_K + 7) / 8), v.n_sub), 256, 0, st>>>(v, d_gexp);
    k_rt_pack<<<dim3((unsigned)((max_K + RT_S - 1) / RT_S), v.n_sub), 256, smem, st>>>(v, d_gexp);
    return cudaGetLastError();
}

// Two launches: the field of every step, the window.
cudaError_t launch_rt_window(const SwrDeviceView& v, cudaStream_t st, const RtPlan& plan, const long long* d_boff,
                             const int* d_win_prev, double* d_theta, int cap, unsigned* d_sweeps, const int* d_gexp,
                             int max_K, int qel, long long spin_limit) {
    RtArgs a;
    a.v = v;
    a.boff = d_boff;
    a.win_prev = d_win_prev;
    a.theta = d_theta;
    a.sweeps = d_sweeps;
    a.gexp = d_gexp;
    a.spin_limit = spin_limit;
    a.cap = cap;
    a.cs = plan.cs;
    a.kmax = max_K;
    a.qel = (qel + 1) & ~1;
    a.nst = plan.nst;
    a.own_smem = plan.own;
    k_rt_theta<<<dim3((unsigned)(cap / 128 + 1), v.n_inst), 128, 0, st>>>(v, d_theta, cap);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cudaError_t e = rt_config(&cfg, at, v.n_sub, plan.cs, rt_smem_bytes(max_K, qel, plan.cs, plan.nst, plan.own != 0));
    if (e != cudaSuccess) return e;
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, k_rt_window, a);
}

}  // namespace swr
