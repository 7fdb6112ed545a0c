// swr_mlp.cu -- small BF16 multilayer perceptron with its own training kernels.
//
// Predicts the initial interface traces of the SWR iteration from subdomain
// descriptors (learned initial guess; not part of the paper's method, which
// starts from g^(0) = 0).  Architecture: n_in -> width -> ... -> width -> n_out,
// tanh after every hidden layer, identity output.  Weights are kept in FP32
// (master copy, Adam moments) and rounded to BF16 for the products; every
// product runs on the 5th-generation tensor cores (tcgen05.mma kind::f16, BF16
// inputs, FP32 accumulation in tensor memory).  Training minimises the mean
// squared error with Adam.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <string>
#include <vector>

#include "swr_internal.cuh"

namespace swr {

// ------------------------------------------------- operand tiles
//
// Every product reads operands that already lie in global memory as the
// shared-memory image the tensor cores take, so that staging a block is one
// contiguous bulk copy (element-wise staging held the products at 25 to 480 us
// each).  A tile of R rows x 64 columns (BF16) is stored as core matrices of
// 8 rows x 16 bytes, row-adjacent cores 128 bytes apart, column-adjacent cores
// 16 R bytes apart; zero outside the matrix.
//   activations, dZ: tiles of 128 batch rows, [row tile][column tile]
//   weights, for Z = H W:     rows = output unit, columns = input unit (64 rows)
//   weights, for dH = dZ W^T: rows = input unit, columns = output unit (64 rows)
// The same activation image serves dW = H^T dZ: there the batch is the
// contraction index and the features the M / N index ("MN-major" operands),
// which exchanges the roles of the two core strides.
#define TC_M 128
#define TC_N 64
#define TC_THREADS 128
#define TC_SPIN (1LL << 22)
#define A_TILE (TC_M * 64 * 2)  // bytes of an activation tile
#define W_TILE (TC_N * 64 * 2)  // bytes of a weight tile
#define FWD_STAGES 4
#define GRAD_STAGES 3
#define FWD_STAGE_BYTES (A_TILE + W_TILE)
#define GRAD_STAGE_BYTES (3 * A_TILE)

__host__ __device__ inline int tiles64(int n) { return (n + 63) >> 6; }
// Byte offset of element (r, c) inside a tile of R rows.
template <int R>
__host__ __device__ inline int tile_off(int r, int c) {
    return (c >> 3) * (16 * R) + (r >> 3) * 128 + (r & 7) * 16 + (c & 7) * 2;
}

__device__ inline unsigned tc_smem(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor without swizzle, version 1.  K-major: lbo =
// bytes between cores adjacent in K, sbo = in M (N); MN-major the same.
__device__ inline unsigned long long tc_desc(unsigned saddr, unsigned lbo, unsigned sbo) {
    unsigned long long d = (unsigned long long)((saddr >> 4) & 0x3FFFu);
    d |= (unsigned long long)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (unsigned long long)((sbo >> 4) & 0x3FFFu) << 32;
    d |= 1ULL << 46;
    return d;
}

__device__ inline bool tc_wait(unsigned mbar, int parity) {
    for (long long it = 0; it < TC_SPIN; ++it) {
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
__device__ inline void tc_bulk(unsigned dst, const void* src, unsigned bytes, unsigned mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}
__device__ inline void tc_mma(unsigned tmem, unsigned long long ad, unsigned long long bd, unsigned idesc, unsigned acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}
__device__ inline void tc_commit(unsigned mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}
// Programmatic dependent launch: a kernel's set-up overlaps the end of the one
// before it; its dependent may start once every CTA here has seen that one's
// results (so everything two kernels back is complete for the dependent).
__device__ inline void pdl_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("fence.proxy.async.global;" ::: "memory");  // bulk copies read what it wrote
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Shared set-up of the product kernels: 64 tensor-memory columns and the ring's
// barriers (full[s], empty[s], done).
struct TcShared {
    unsigned long long full[4], empty[4], done;
    unsigned tmem_slot;
    int fail;
};
__device__ inline unsigned tc_begin(TcShared& sh) {
    if ((threadIdx.x >> 5) == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(&sh.tmem_slot)),
                     "r"(TC_N));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        for (int i = 0; i < 4; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&sh.full[i])));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&sh.empty[i])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&sh.done)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sh.fail = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    return sh.tmem_slot;
}

// The ring: warp 0 lane 0 fills stages (load(stage address, block, barrier) issues
// `bytes` of bulk copies), warp 1 lane 0 issues the block's products
// (mma(stage address, block)) and frees the stage on their completion.  Every
// thread then waits for the last product.  All waits are bounded; a thread that
// gives up records it, the others run into their own limit or the done
// barrier, and then the copies issued last into every stage are waited for,
// whichever thread gave up: a CTA must not return while one still writes its
// shared memory.
template <int STAGES, class Load, class Mma>
__device__ inline bool tc_pipeline(TcShared& sh, unsigned char* ring, int stage_bytes, int nblk, unsigned bytes, Load load,
                                   Mma mma) {
    int issued = 0;
    if (threadIdx.x == 0) {
        bool ok = true;
        for (int b = 0; b < nblk && ok; ++b) {
            const int st = b % STAGES;
            if (b >= STAGES) ok = tc_wait(tc_smem(&sh.empty[st]), ((b / STAGES) & 1) ^ 1);
            if (!ok) break;
            const unsigned bar = tc_smem(&sh.full[st]);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
            load(tc_smem(ring + (size_t)st * stage_bytes), b, bar);
            issued = b + 1;
        }
        if (!ok) sh.fail = 1;
    } else if (threadIdx.x == 32) {
        bool ok = true;
        for (int b = 0; b < nblk && ok; ++b) {
            const int st = b % STAGES;
            ok = tc_wait(tc_smem(&sh.full[st]), (b / STAGES) & 1);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            mma(tc_smem(ring + (size_t)st * stage_bytes), b);
            tc_commit(tc_smem(&sh.empty[st]));
        }
        if (!ok) sh.fail = 1;
        tc_commit(tc_smem(&sh.done));
    }
    __syncwarp();
    if (!tc_wait(tc_smem(&sh.done), 0)) sh.fail = 1;
    __syncthreads();
    if (sh.fail && threadIdx.x == 0)
        for (int b = issued > STAGES ? issued - STAGES : 0; b < issued; ++b)
            tc_wait(tc_smem(&sh.full[b % STAGES]), (b / STAGES) & 1);
    asm volatile("tcgen05.fence::after_thread_sync;");
    return sh.fail == 0;
}
__device__ inline void tc_end(unsigned tmem) {
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if ((threadIdx.x >> 5) == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_N));
}
__device__ inline void tc_ld16(unsigned tmem, int c0, float (&v)[16]) {
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(tmem + ((unsigned)((threadIdx.x >> 5) * 32) << 16) + (unsigned)c0));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// kind::f16 instruction descriptor: D F32, A and B BF16; mn = 1: both operands
// MN-major.
__device__ inline unsigned tc_idesc(int mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)mn << 15) | ((unsigned)mn << 16) |
           ((unsigned)(TC_N >> 3) << 17) | ((unsigned)(TC_M >> 4) << 24);
}

// Sixteen columns of one row into a 128-row tile (BF16), zero past the batch.
__device__ inline void store_tile16(unsigned char* tile, int row, int c0, const float (&h)[16]) {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        unsigned w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(h[8 * g + 2 * j], h[8 * g + 2 * j + 1]);
            w[j] = *reinterpret_cast<const unsigned*>(&p);
        }
        *reinterpret_cast<uint4*>(tile + tile_off<TC_M>(row, c0 + 8 * g)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Sixteen columns of a row of an FP32 matrix with `n` columns (at most `left`
// of them inside it); 16-byte accesses where the row allows it.
__device__ inline bool row_vec(const float* p, int n, int left) { return left >= 16 && !(n & 3) && !((size_t)p & 15); }
__device__ inline void row_store16(float* p, int n, int left, const float (&z)[16]) {
    if (row_vec(p, n, left)) {
#pragma unroll
        for (int j = 0; j < 16; j += 4) *reinterpret_cast<float4*>(p + j) = make_float4(z[j], z[j + 1], z[j + 2], z[j + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j < left) p[j] = z[j];
    }
}
__device__ inline void row_load16(const float* p, int n, int left, float (&z)[16]) {
    if (row_vec(p, n, left)) {
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
            const float4 q = *reinterpret_cast<const float4*>(p + j);
            z[j] = q.x;
            z[j + 1] = q.y;
            z[j + 2] = q.z;
            z[j + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) z[j] = j < left ? p[j] : 0.f;
    }
}

enum MlpEpilogue { EP_HIDDEN = 0, EP_OUT = 1, EP_MSE = 2, EP_BACK = 3 };
struct MlpLayer {
    const unsigned char* A;   // activation tiles [row tile][ka] of the product's left operand
    const unsigned char* W;   // weight tiles [column tile][ka]
    unsigned char* out_t;     // EP_HIDDEN, EP_MSE, EP_BACK: BF16 tiles of the result [row tile][tiles64(N)]
    float* out_f;             // EP_HIDDEN: tanh values (training only, else null); EP_OUT: y; else dZ in FP32
                              // with tiles64(N) * 64 columns
    const float* bias;        // EP_HIDDEN, EP_OUT, EP_MSE
    const float* other;       // EP_MSE: target t; EP_BACK: tanh values of the layer
    float* loss;              // EP_MSE: [row tile][column tile] sums of squares
    float scale;              // EP_MSE: 2 / (batch N)
    int batch, N, ka;
};

// One product C = A W (128 x 64 tile of C per CTA, contraction ka x 64) with its
// layer's epilogue: bias and tanh into the next operand's tiles (EP_HIDDEN),
// the output (EP_OUT), the squared error with its gradient (EP_MSE), or the
// chain through tanh for dH = dZ W^T (EP_BACK).  Latency bound at these sizes
// (4 products of width 256): blocks stream through a 4-stage bulk-copy ring,
// and the separate bias / tanh / error / conversion passes and copies are
// gone.  Per launch at width 256 (cold caches): 9 us at a batch of 16 (25 + 3
// before), 11 us at 2560 (47 + 11 before; the back-propagation 109 + 5);
// whole calls: forward of 16 rows 127 -> 50 us, training step of 2560 rows
// with its gradient read back 1859 -> 133 us.
template <int EP>
__global__ void __launch_bounds__(TC_THREADS) k_mlp_layer(MlpLayer p, volatile int* err) {
    extern __shared__ __align__(1024) unsigned char ring[];
    __shared__ TcShared sh;
    __shared__ float s_red[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int mt = blockIdx.y, nt = blockIdx.x;
    const unsigned tmem = tc_begin(sh);
    pdl_wait();
    const unsigned idesc = tc_idesc(0);
    const bool ok = tc_pipeline<FWD_STAGES>(
        sh, ring, FWD_STAGE_BYTES, p.ka, FWD_STAGE_BYTES,
        [&](unsigned dst, int b, unsigned bar) {
            tc_bulk(dst, p.A + ((size_t)mt * p.ka + b) * A_TILE, A_TILE, bar);
            tc_bulk(dst + A_TILE, p.W + ((size_t)nt * p.ka + b) * W_TILE, W_TILE, bar);
        },
        [&](unsigned src, int b) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                tc_mma(tmem, tc_desc(src + kk * 2 * 16 * TC_M, 16 * TC_M, 128),
                       tc_desc(src + A_TILE + kk * 2 * 16 * TC_N, 16 * TC_N, 128), idesc, (b | kk) ? 1u : 0u);
        });
    if (!ok) {
        if (threadIdx.x == 0) *err = 1;
    } else {
        const int r = warp * 32 + lane, row = mt * TC_M + r;
        const bool in = row < p.batch;
        float lsum = 0.f;
#pragma unroll 1
        for (int c0 = 0; c0 < TC_N; c0 += 16) {
            float z[16];
            tc_ld16(tmem, c0, z);
            const int col0 = nt * TC_N + c0;
            if (EP != EP_BACK) {
#pragma unroll
                for (int j = 0; j < 16; ++j) z[j] += col0 + j < p.N ? p.bias[col0 + j] : 0.f;
            }
            if (EP == EP_HIDDEN) {
#pragma unroll
                for (int j = 0; j < 16; ++j) z[j] = in && col0 + j < p.N ? tanhf(z[j]) : 0.f;
                store_tile16(p.out_t + ((size_t)mt * tiles64(p.N) + nt) * A_TILE, r, c0, z);
                if (p.out_f && in) row_store16(p.out_f + (size_t)row * p.N + col0, p.N, p.N - col0, z);
            } else if (EP == EP_OUT) {
                if (in) row_store16(p.out_f + (size_t)row * p.N + col0, p.N, p.N - col0, z);
            } else {
                float o[16];
                row_load16(p.other + (size_t)(in ? row : 0) * p.N + col0, p.N, p.N - col0, o);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const bool ok2 = in && col0 + j < p.N;
                    const float x = o[j];
                    if (EP == EP_MSE) {
                        const float df = z[j] - x;
                        lsum += ok2 ? df * df : 0.f;
                        z[j] = ok2 ? p.scale * df : 0.f;
                    } else {
                        z[j] = ok2 ? z[j] * (1.f - x * x) : 0.f;
                    }
                }
                store_tile16(p.out_t + ((size_t)mt * tiles64(p.N) + nt) * A_TILE, r, c0, z);
                if (in) row_store16(p.out_f + (size_t)row * (tiles64(p.N) * 64) + col0, 64, 16, z);
            }
        }
        if (EP == EP_MSE) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
            if (lane == 0) s_red[warp] = lsum;
            __syncthreads();
            if (threadIdx.x == 0) p.loss[mt * gridDim.x + nt] = (s_red[0] + s_red[1]) + (s_red[2] + s_red[3]);
        }
    }
    tc_end(tmem);
}

// Gradients of every layer in one launch.  CTAs below n_tiles: dW_l = H_l^T
// dZ_l, one 128 x 64 tile each; both operands are the activations' own tiles,
// read MN-major (contraction over the batch, 128 rows a block).  The others:
// db_l = column sums of dZ_l, 32 columns each.  Either sum runs over the batch
// in order in one FP32 accumulator (what the tensor core and one thread per
// column make of it): splitting the batch would fill more SMs, but another
// rounding of near-zero gradients changes the sign-like first Adam steps and so
// the training trajectory.  Bulk copies keep the single chain short: at a
// batch of 2560 (width 256, 1024 outputs) this launch takes about 20 us, the
// element-wise staged products and the unstaged column sums took 2.5 ms.
struct MlpGradJob {
    const unsigned char *H, *Z;  // tiles [row tile][kh], [row tile][kz]
    const float* dz;             // dZ in FP32, kz * 64 columns
    long long w_off, b_off;      // of dW_l and db_l in the parameter vector
    int din, dout, kh, kz, tile0, ntn, col0;  // tile0, col0: first CTA of the layer's tiles, column sums
};
#define COLSUM_ROWS 128
#define COLSUM_STAGES 6
__device__ inline void mlp_colsum(const MlpGradJob& J, int chunk, int batch, float* ring, float* g) {
    const int ld = J.kz * 64, c0 = chunk * 32, nst = (batch + COLSUM_ROWS - 1) / COLSUM_ROWS;
    auto issue = [&](int st) {
        float* dst = ring + (size_t)(st % COLSUM_STAGES) * COLSUM_ROWS * 32;
        if (st < nst)
            for (int e = threadIdx.x; e < COLSUM_ROWS * 8; e += TC_THREADS) {
                const int r = st * COLSUM_ROWS + (e >> 3);
                if (r < batch)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc_smem(dst + (e >> 3) * 32 + (e & 7) * 4)),
                                 "l"(J.dz + (size_t)r * ld + c0 + (e & 7) * 4)
                                 : "memory");
            }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int st = 0; st < COLSUM_STAGES - 1; ++st) issue(st);
    float acc = 0.f;
    for (int st = 0; st < nst; ++st) {
        asm volatile("cp.async.wait_group %0;" ::"n"(COLSUM_STAGES - 2) : "memory");
        __syncthreads();  // stage st is complete, and the stage refilled next has been summed
        issue(st + COLSUM_STAGES - 1);
        if (threadIdx.x < 32) {
            const float* src = ring + (size_t)(st % COLSUM_STAGES) * COLSUM_ROWS * 32 + threadIdx.x;
            const int rows = min(COLSUM_ROWS, batch - st * COLSUM_ROWS);
#pragma unroll 16
            for (int r = 0; r < rows; ++r) acc += src[r * 32];
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (threadIdx.x < 32 && c0 + (int)threadIdx.x < J.dout) g[J.b_off + c0 + threadIdx.x] = acc;
}

__global__ void __launch_bounds__(TC_THREADS) k_mlp_grad(const MlpGradJob* jobs, int n_jobs, int n_tiles, int batch,
                                                         float* g, volatile int* err) {
    extern __shared__ __align__(1024) unsigned char ring[];
    __shared__ TcShared sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int l = 0;
    if ((int)blockIdx.x >= n_tiles) {
        pdl_wait();
        const int c = blockIdx.x - n_tiles;
        while (l + 1 < n_jobs && c >= jobs[l + 1].col0) ++l;
        mlp_colsum(jobs[l], c - jobs[l].col0, batch, reinterpret_cast<float*>(ring), g);
        return;
    }
    const unsigned tmem = tc_begin(sh);
    pdl_wait();
    while (l + 1 < n_jobs && (int)blockIdx.x >= jobs[l + 1].tile0) ++l;
    const MlpGradJob J = jobs[l];
    const int t = blockIdx.x - J.tile0, ti = t / J.ntn, tj = t - ti * J.ntn;
    const int np = min(2, J.kh - 2 * ti);  // 64-feature tiles of H under this 128-row tile
    const unsigned idesc = tc_idesc(1);
    const bool ok = tc_pipeline<GRAD_STAGES>(
        sh, ring, GRAD_STAGE_BYTES, (batch + TC_M - 1) / TC_M, (unsigned)(np + 1) * A_TILE,
        [&](unsigned dst, int b, unsigned bar) {
            for (int u = 0; u < np; ++u)
                tc_bulk(dst + u * A_TILE, J.H + ((size_t)b * J.kh + 2 * ti + u) * A_TILE, A_TILE, bar);
            tc_bulk(dst + 2 * A_TILE, J.Z + ((size_t)b * J.kz + tj) * A_TILE, A_TILE, bar);
        },
        [&](unsigned src, int b) {
            // rows of the tile past np x 64 take whatever the stage holds: they are not stored
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                tc_mma(tmem, tc_desc(src + kk * 256, 128, 16 * TC_M),
                       tc_desc(src + 2 * A_TILE + kk * 256, 128, 16 * TC_M), idesc, (b | kk) ? 1u : 0u);
        });
    if (!ok) {
        if (threadIdx.x == 0) *err = 1;
    } else {
        const int row = ti * TC_M + warp * 32 + lane;
#pragma unroll 1
        for (int c0 = 0; c0 < TC_N; c0 += 16) {
            float z[16];
            tc_ld16(tmem, c0, z);
            const int col0 = tj * TC_N + c0;
            if (row < J.din) row_store16(g + J.w_off + (size_t)row * J.dout + col0, J.dout, J.dout - col0, z);
        }
    }
    tc_end(tmem);
}

// x [batch x n] FP32 -> BF16 tiles, zero outside.
__global__ void k_mlp_pack(const float* x, unsigned char* tiles, int batch, int n, int mtiles) {
    pdl_wait();
    const int kt = tiles64(n);
    const long long total = (long long)mtiles * TC_M * kt * 8;  // groups of 8 columns
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int g = (int)(e % (kt * 8)), row = (int)(e / (kt * 8));
        unsigned w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = g * 8 + 2 * j;
            const float a = row < batch && c < n ? x[(size_t)row * n + c] : 0.f;
            const float b = row < batch && c + 1 < n ? x[(size_t)row * n + c + 1] : 0.f;
            const __nv_bfloat162 q = __floats2bfloat162_rn(a, b);
            w[j] = *reinterpret_cast<const unsigned*>(&q);
        }
        *reinterpret_cast<uint4*>(tiles + ((size_t)(row / TC_M) * kt + (g >> 3)) * A_TILE +
                                  tile_off<TC_M>(row % TC_M, (g & 7) * 8)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Layer blockIdx.y: one Adam step on the FP32 parameters (adam) and the BF16
// weight tiles of their values.
struct MlpParamLayer {
    long long w_off;          // the layer's weights, followed by its biases
    unsigned char *wf, *wt;   // tiles for Z = H W and dH = dZ W^T
    int din, dout;
};
__global__ void k_mlp_params(const MlpParamLayer* layers, float* p, const float* g, float* m, float* v, int adam, float lr,
                             float b1, float b2, float eps, float c1, float c2) {
    pdl_wait();
    const MlpParamLayer L = layers[blockIdx.y];
    const long long nw = (long long)L.din * L.dout, n = nw + L.dout;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        const long long e = L.w_off + q;
        float x = p[e];
        if (adam) {
            const float gr = g[e];
            const float mm = b1 * m[e] + (1.f - b1) * gr, vv = b2 * v[e] + (1.f - b2) * gr * gr;
            m[e] = mm;
            v[e] = vv;
            x -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
            p[e] = x;
        }
        if (q < nw) {
            const int r = (int)(q / L.dout), c = (int)(q - (long long)r * L.dout);
            const __nv_bfloat16 h = __float2bfloat16(x);
            *reinterpret_cast<__nv_bfloat16*>(L.wf + ((size_t)(c >> 6) * tiles64(L.din) + (r >> 6)) * W_TILE +
                                              tile_off<TC_N>(c & 63, r & 63)) = h;
            *reinterpret_cast<__nv_bfloat16*>(L.wt + ((size_t)(r >> 6) * tiles64(L.dout) + (c >> 6)) * W_TILE +
                                              tile_off<TC_N>(r & 63, c & 63)) = h;
        }
    }
}

}  // namespace swr

using namespace swr;

struct swr_mlp {
    std::string err;
    int n_in, width, n_hidden, n_out, n_layers;
    std::vector<int> dims;             // n_layers + 1
    std::vector<long long> w_off, b_off;  // into the parameter vector
    long long n_params = 0;
    cudaStream_t stream = nullptr;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // params, grads, Adam moments
    unsigned char* wtiles = nullptr;   // BF16 weight tiles of every layer, both orientations
    std::vector<unsigned char*> wf, wt;
    int cap_batch = 0;
    char* work = nullptr;              // activations of a batch (one allocation)
    std::vector<unsigned char*> act;   // per layer input: BF16 tiles (layer 0: x)
    std::vector<unsigned char*> dz;    // per layer output: BF16 tiles of dZ
    std::vector<float*> hf, dzf;       // per layer output: tanh values, dZ in FP32
    MlpGradJob* d_jobs = nullptr;
    MlpParamLayer* d_layers = nullptr;
    int n_grad_tiles = 0, n_colsum = 0;
    volatile int* flag = nullptr;      // host-mapped: set by a product whose completion wait timed out
    int* d_flag = nullptr;
    float *h_loss = nullptr, *d_loss = nullptr;  // host-mapped loss partials
    size_t h_loss_n = 0;
    long long adam_t = 0;
};

static swr_status mlp_fail(swr_mlp* m, swr_status s, const char* msg) {
    if (m) m->err = msg;
    return s;
}

#define MCU(call)                                                         \
    do {                                                                  \
        cudaError_t e_ = (call);                                          \
        if (e_ != cudaSuccess) return mlp_fail(m, SWR_ECUDA, cudaGetErrorString(e_)); \
    } while (0)

static unsigned gsz(long long n) { return (unsigned)(n < 256LL * 4096 ? (n + 255) / 256 : 4096); }

// Launch with programmatic dependent launch (the kernels begin with pdl_wait).
template <class... KArgs, class... Args>
static cudaError_t launch_pdl(void (*k)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, KArgs(args)...);
}

static int row_tiles(int batch) { return (batch + TC_M - 1) / TC_M; }

// Buffers for a batch, in one allocation kept until a larger batch comes.
static swr_status ensure_batch(swr_mlp* m, int batch) {
    if (batch <= m->cap_batch) return SWR_OK;
    MCU(cudaStreamSynchronize(m->stream));
    cudaFree(m->work);
    m->work = nullptr;
    m->cap_batch = 0;
    const int L = m->n_layers;
    const size_t mt = (size_t)row_tiles(batch);
    size_t used = 0;
    auto add = [&](size_t bytes) {
        const size_t o = used;
        used += (bytes + 255) & ~(size_t)255;
        return o;
    };
    std::vector<size_t> oa(L), oz(L), oh(L), oc(L);
    for (int l = 0; l < L; ++l) {
        oa[l] = add(mt * tiles64(m->dims[l]) * A_TILE);
        oz[l] = add(mt * tiles64(m->dims[l + 1]) * A_TILE);
        oh[l] = add(sizeof(float) * (size_t)batch * m->dims[l + 1]);
        oc[l] = add(sizeof(float) * (size_t)batch * tiles64(m->dims[l + 1]) * 64);
    }
    const size_t nloss = mt * tiles64(m->n_out);
    std::vector<MlpGradJob> jobs(L);
    int tiles = 0, cols = 0;
    for (int l = 0; l < L; ++l) {
        jobs[l].din = m->dims[l];
        jobs[l].dout = m->dims[l + 1];
        jobs[l].kh = tiles64(m->dims[l]);
        jobs[l].kz = tiles64(m->dims[l + 1]);
        jobs[l].w_off = m->w_off[l];
        jobs[l].b_off = m->b_off[l];
        jobs[l].tile0 = tiles;
        jobs[l].col0 = cols;
        jobs[l].ntn = jobs[l].kz;
        cols += (m->dims[l + 1] + 31) / 32;
        tiles += (m->dims[l] + TC_M - 1) / TC_M * jobs[l].ntn;
    }
    if (cudaMalloc((void**)&m->work, used) != cudaSuccess) {
        cudaGetLastError();
        m->work = nullptr;
        return mlp_fail(m, SWR_ECUDA, "out of memory");
    }
    if (nloss > m->h_loss_n) {
        cudaFreeHost(m->h_loss);
        m->h_loss = nullptr;
        m->h_loss_n = 0;
        MCU(cudaHostAlloc((void**)&m->h_loss, sizeof(float) * nloss, cudaHostAllocMapped));
        MCU(cudaHostGetDevicePointer((void**)&m->d_loss, m->h_loss, 0));
        m->h_loss_n = nloss;
    }
    m->act.resize(L);
    m->dz.resize(L);
    m->hf.resize(L);
    m->dzf.resize(L);
    for (int l = 0; l < L; ++l) {
        m->act[l] = (unsigned char*)m->work + oa[l];
        m->dz[l] = (unsigned char*)m->work + oz[l];
        m->hf[l] = (float*)(m->work + oh[l]);
        m->dzf[l] = (float*)(m->work + oc[l]);
        jobs[l].H = m->act[l];
        jobs[l].Z = m->dz[l];
        jobs[l].dz = m->dzf[l];
    }
    m->n_grad_tiles = tiles;
    m->n_colsum = cols;
    MCU(cudaMemcpyAsync(m->d_jobs, jobs.data(), sizeof(MlpGradJob) * L, cudaMemcpyHostToDevice, m->stream));
    MCU(cudaStreamSynchronize(m->stream));
    m->cap_batch = batch;
    return SWR_OK;
}

// Waits for the stream and reads the tensor-core timeout flag.
static swr_status finish(swr_mlp* m) {
    MCU(cudaStreamSynchronize(m->stream));
    if (*m->flag) return mlp_fail(m, SWR_ETIMEOUT, "a tensor-core product did not complete (bounded wait)");
    return SWR_OK;
}

// BF16 weight tiles from the FP32 parameters (no gradient, no update).
static cudaError_t refresh_tiles(swr_mlp* m) {
    return launch_pdl(k_mlp_params, dim3(256, m->n_layers), 256, 0, m->stream, m->d_layers, m->p, m->g, m->m, m->v, 0, 0.f,
                      0.f, 0.f, 0.f, 1.f, 1.f);
}

extern "C" swr_status swr_mlp_create(int n_in, int width, int n_hidden, int n_out, void* stream, swr_mlp** out) {
    if (!out || n_in < 1 || width < 1 || n_hidden < 1 || n_out < 1 || n_in > 65536 || width > 65536 || n_out > 65536)
        return SWR_EINVAL;
    swr_mlp* m = new swr_mlp();
    m->n_in = n_in;
    m->width = width;
    m->n_hidden = n_hidden;
    m->n_out = n_out;
    m->n_layers = n_hidden + 1;
    m->stream = (cudaStream_t)stream;
    m->dims.push_back(n_in);
    for (int i = 0; i < n_hidden; ++i) m->dims.push_back(width);
    m->dims.push_back(n_out);
    long long off = 0;
    size_t tb = 0;
    std::vector<size_t> of(m->n_layers), ot(m->n_layers);
    for (int l = 0; l < m->n_layers; ++l) {
        m->w_off.push_back(off);
        off += (long long)m->dims[l] * m->dims[l + 1];
        m->b_off.push_back(off);
        off += m->dims[l + 1];
        const size_t bytes = (size_t)tiles64(m->dims[l]) * tiles64(m->dims[l + 1]) * W_TILE;
        of[l] = tb;
        ot[l] = tb + bytes;
        tb += 2 * bytes;
    }
    m->n_params = off;
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = cudaMalloc(&m->p, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMalloc(&m->g, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMalloc(&m->m, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMalloc(&m->v, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMalloc(&m->wtiles, tb);
    if (e == cudaSuccess) e = cudaMalloc(&m->d_jobs, sizeof(MlpGradJob) * m->n_layers);
    if (e == cudaSuccess) e = cudaMalloc(&m->d_layers, sizeof(MlpParamLayer) * m->n_layers);
    if (e == cudaSuccess) e = cudaHostAlloc((void**)&m->flag, sizeof(int), cudaHostAllocMapped);
    if (e == cudaSuccess) {
        *m->flag = 0;
        e = cudaHostGetDevicePointer((void**)&m->d_flag, (void*)m->flag, 0);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(m->m, 0, sizeof(float) * off, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->v, 0, sizeof(float) * off, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->p, 0, sizeof(float) * off, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->wtiles, 0, tb, m->stream);  // zero parameters, zero padding
    if (e == cudaSuccess) {
        const int fs = FWD_STAGES * FWD_STAGE_BYTES, gs = GRAD_STAGES * GRAD_STAGE_BYTES;
        const void* f[4] = {(const void*)k_mlp_layer<EP_HIDDEN>, (const void*)k_mlp_layer<EP_OUT>,
                            (const void*)k_mlp_layer<EP_MSE>, (const void*)k_mlp_layer<EP_BACK>};
        for (int i = 0; i < 4 && e == cudaSuccess; ++i)
            e = cudaFuncSetAttribute(f[i], cudaFuncAttributeMaxDynamicSharedMemorySize, fs);
        if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, gs);
    }
    if (e == cudaSuccess) {
        std::vector<MlpParamLayer> pl;
        for (int l = 0; l < m->n_layers; ++l) {
            m->wf.push_back(m->wtiles + of[l]);
            m->wt.push_back(m->wtiles + ot[l]);
            MlpParamLayer q;
            q.w_off = m->w_off[l];
            q.wf = m->wf[l];
            q.wt = m->wt[l];
            q.din = m->dims[l];
            q.dout = m->dims[l + 1];
            pl.push_back(q);
        }
        e = cudaMemcpyAsync(m->d_layers, pl.data(), sizeof(MlpParamLayer) * pl.size(), cudaMemcpyHostToDevice, m->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        swr_mlp_destroy(m);
        return SWR_ENOMEM;
    }
    *out = m;
    return SWR_OK;
}

extern "C" swr_status swr_mlp_param_count(swr_mlp* m, size_t* n) {
    if (!m || !n) return SWR_EINVAL;
    *n = (size_t)m->n_params;
    return SWR_OK;
}

extern "C" swr_status swr_mlp_set_params(swr_mlp* m, const float* host, size_t n) {
    if (!m || !host || n != (size_t)m->n_params) return mlp_fail(m, SWR_EINVAL, "parameter count mismatch");
    MCU(cudaMemcpyAsync(m->p, host, sizeof(float) * n, cudaMemcpyHostToDevice, m->stream));
    MCU(cudaMemsetAsync(m->m, 0, sizeof(float) * n, m->stream));
    MCU(cudaMemsetAsync(m->v, 0, sizeof(float) * n, m->stream));
    m->adam_t = 0;
    MCU(refresh_tiles(m));
    MCU(cudaStreamSynchronize(m->stream));
    return SWR_OK;
}

extern "C" swr_status swr_mlp_get_params(swr_mlp* m, float* host, size_t n) {
    if (!m || !host || n != (size_t)m->n_params) return mlp_fail(m, SWR_EINVAL, "parameter count mismatch");
    MCU(cudaMemcpyAsync(host, m->p, sizeof(float) * n, cudaMemcpyDeviceToHost, m->stream));
    MCU(cudaStreamSynchronize(m->stream));
    return SWR_OK;
}

// Hidden layers and the last product on device arrays: x [batch x n_in] FP32;
// y: the output (inference), t: the target (training: error and dZ of the
// output layer instead of y).
static swr_status forward(swr_mlp* m, const float* x, int batch, float* y, const float* t) {
    swr_status st = ensure_batch(m, batch);
    if (st != SWR_OK) return st;
    cudaStream_t s = m->stream;
    const int mt = row_tiles(batch);
    MCU(launch_pdl(k_mlp_pack, dim3(gsz((long long)mt * TC_M * tiles64(m->n_in) * 8)), 256, 0, s, x, m->act[0], batch,
                   m->n_in, mt));
    for (int l = 0; l < m->n_layers; ++l) {
        const bool last = l == m->n_layers - 1;
        MlpLayer a;
        memset(&a, 0, sizeof(a));
        a.A = m->act[l];
        a.W = m->wf[l];
        a.bias = m->p + m->b_off[l];
        a.batch = batch;
        a.N = m->dims[l + 1];
        a.ka = tiles64(m->dims[l]);
        const dim3 grid(tiles64(a.N), mt);
        const size_t sm = FWD_STAGES * FWD_STAGE_BYTES;
        if (!last) {
            a.out_t = m->act[l + 1];
            a.out_f = t ? m->hf[l] : nullptr;
            MCU(launch_pdl(k_mlp_layer<EP_HIDDEN>, grid, TC_THREADS, sm, s, a, m->d_flag));
        } else if (!t) {
            a.out_f = y;
            MCU(launch_pdl(k_mlp_layer<EP_OUT>, grid, TC_THREADS, sm, s, a, m->d_flag));
        } else {
            a.out_t = m->dz[l];
            a.other = t;
            a.out_f = m->dzf[l];
            a.loss = m->d_loss;
            a.scale = 2.f / (float)((long long)batch * m->n_out);
            MCU(launch_pdl(k_mlp_layer<EP_MSE>, grid, TC_THREADS, sm, s, a, m->d_flag));
        }
    }
    return SWR_OK;
}

extern "C" swr_status swr_mlp_forward(swr_mlp* m, const float* x_dev, int batch, float* y_dev) {
    if (!m || !x_dev || !y_dev || batch < 1) return mlp_fail(m, SWR_EINVAL, "bad argument");
    swr_status st = forward(m, x_dev, batch, y_dev, nullptr);
    if (st != SWR_OK) return st;
    MCU(cudaGetLastError());
    return finish(m);
}

// One Adam step on the mean squared error; loss_host (nullable) receives the
// loss before the update, grad_host (nullable) the gradient (n_params floats).
extern "C" swr_status swr_mlp_train_step(swr_mlp* m, const float* x_dev, const float* t_dev, int batch, float lr,
                                         float* loss_host, float* grad_host) {
    if (!m || !x_dev || !t_dev || batch < 1) return mlp_fail(m, SWR_EINVAL, "bad argument");
    swr_status st = forward(m, x_dev, batch, nullptr, t_dev);
    if (st != SWR_OK) return st;
    cudaStream_t s = m->stream;
    const int L = m->n_layers, mt = row_tiles(batch);
    const size_t nloss = (size_t)mt * tiles64(m->n_out);
    for (int l = L - 1; l > 0; --l) {
        // dZ of layer l - 1 = (dZ_l W_l^T) (1 - h^2)
        MlpLayer a;
        memset(&a, 0, sizeof(a));
        a.A = m->dz[l];
        a.W = m->wt[l];
        a.out_t = m->dz[l - 1];
        a.other = m->hf[l - 1];
        a.out_f = m->dzf[l - 1];
        a.batch = batch;
        a.N = m->dims[l];
        a.ka = tiles64(m->dims[l + 1]);
        MCU(launch_pdl(k_mlp_layer<EP_BACK>, dim3(tiles64(a.N), mt), TC_THREADS, (size_t)FWD_STAGES * FWD_STAGE_BYTES, s, a,
                       m->d_flag));
    }
    MCU(launch_pdl(k_mlp_grad, dim3(m->n_grad_tiles + m->n_colsum), TC_THREADS, (size_t)GRAD_STAGES * GRAD_STAGE_BYTES, s,
                   m->d_jobs, L, m->n_grad_tiles, batch, m->g, m->d_flag));
    if (lr > 0.f) {
        m->adam_t += 1;
        const float b1 = 0.9f, b2 = 0.999f;
        const float c1 = 1.f - powf(b1, (float)m->adam_t), c2 = 1.f - powf(b2, (float)m->adam_t);
        MCU(launch_pdl(k_mlp_params, dim3(256, L), 256, 0, s, m->d_layers, m->p, m->g, m->m, m->v, 1, lr, b1, b2, 1e-8f, c1,
                       c2));
    }
    if (grad_host) MCU(cudaMemcpyAsync(grad_host, m->g, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost, s));
    MCU(cudaGetLastError());
    st = finish(m);
    if (st != SWR_OK) return st;
    if (loss_host) {
        double acc = 0;
        for (size_t i = 0; i < nloss; ++i) acc += m->h_loss[i];
        *loss_host = (float)(acc / (double)((long long)batch * m->n_out));
    }
    return SWR_OK;
}

extern "C" void swr_mlp_destroy(swr_mlp* m) {
    if (!m) return;
    if (m->stream) cudaStreamSynchronize(m->stream);
    cudaFree(m->work);
    cudaFree(m->p);
    cudaFree(m->g);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->wtiles);
    cudaFree(m->d_jobs);
    cudaFree(m->d_layers);
    if (m->flag) cudaFreeHost((void*)m->flag);
    cudaFreeHost(m->h_loss);
    delete m;
}

extern "C" const char* swr_mlp_last_error(const swr_mlp* m) { return m ? m->err.c_str() : ""; }
