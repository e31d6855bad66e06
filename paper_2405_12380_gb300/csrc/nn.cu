// Dense layers of the DeepONet (App. B): FP32 GEMM, bias + activation and their
// gradients, the relative-L2 loss of the DeepONet output, and Adam.
//
// Row-major matrices throughout.  Long-K products of the GEMM are split over
// blockIdx.z and combined with atomic adds (training tolerates the summation order).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "helm_internal.cuh"

namespace {

// ---- FP32 GEMM: C += alpha op(A) op(B) over a slice of K (blockIdx.z)
//
// A block of (BM / 8)(BN / 8) threads owns a BM x BN tile of C, 8 x 8 per thread; a warp
// covers 32 x 64 of it (4 x 8 threads), so that one K step of a warp reads four 128-byte
// wavefronts of shared memory for 64 FMA instructions per scheduler.  Slabs of SBK K
// values of both operands are held K-major in two shared buffers; the next slab's global
// loads are issued before the current one is used, 16 bytes per thread where the operand
// allows it (VA / VB: leading dimension a multiple of 4 and a 16-byte aligned base).
// Bound by the FP32 pipe for square products (16384 x 256 x 256: 93 -> 30 us, 72 of the
// pipe's 80 TFLOP/s), by the FP32 pipe and HBM about equally for the branch's first layer
// at 64^3 (32 x 256 x 524288, 537 MB of weights read: 1060 -> 206 us; its weight gradient,
// 537 MB written: 842 -> 181 us).  Before: 64 x 64 tiles, 4 x 4 per thread, 4-byte loads,
// no prefetch, and 64-row tiles half empty at a batch of 32.  The packed fma.rn.f32x2
// issues two multiply-adds per instruction.
constexpr int SBK = 16;

__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
    return v;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
// two FP32 fused multiply-adds in one instruction (each rounded as fmaf)
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// one SBK x R slab of an operand, global -> registers -> shared [SBK][R + 4].
// KC: stored with K contiguous (element (r, k) at X[r ld + k]); else (r, k) at X[k ld + r]
template <int R, int T, bool KC>
struct Slab {
    static constexpr int Q = R * SBK / 4 / T;              // groups of four values per thread
    static_assert(Q * T * 4 == R * SBK, "the slab divides among the threads");
    float4 v[Q];

    __device__ __forceinline__ void load(const float* __restrict__ X, long long ld, int r0, int rows, int k0, int k1,
                                         bool vec) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int t = threadIdx.x + q * T;
            const int r = KC ? t / (SBK / 4) : (t % (R / 4)) * 4, k = KC ? (t % (SBK / 4)) * 4 : t / (R / 4);
            const int gr = r0 + r, gk = k0 + k;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            const int n = KC ? (gr < rows ? k1 - gk : 0) : (gk < k1 ? rows - gr : 0);   // values that exist
            const float* p = X + (KC ? (long long)gr * ld + gk : (long long)gk * ld + gr);
            if (n >= 4 && vec) {
                x = __ldg(reinterpret_cast<const float4*>(p));
            } else if (n > 0) {
                x.x = __ldg(p);
                if (n > 1) x.y = __ldg(p + 1);
                if (n > 2) x.z = __ldg(p + 2);
                if (n > 3) x.w = __ldg(p + 3);
            }
            v[q] = x;
        }
    }
    __device__ __forceinline__ void store(float (*S)[R + 4]) const {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int t = threadIdx.x + q * T;
            if (KC) {
                const int r = t / (SBK / 4), k = (t % (SBK / 4)) * 4;
                S[k][r] = v[q].x;
                S[k + 1][r] = v[q].y;
                S[k + 2][r] = v[q].z;
                S[k + 3][r] = v[q].w;
            } else {
                *reinterpret_cast<float4*>(&S[t / (R / 4)][(t % (R / 4)) * 4]) = v[q];
            }
        }
    }
};

template <int BM, int BN, bool AKC, bool BKC>
__global__ void __launch_bounds__(BM * BN / 64, BM * BN / 64 >= 256 ? 2 : 3)
    k_sgemm(int M, int N, int K, float alpha, const float* __restrict__ A, int lda, const float* __restrict__ B,
            int ldb, float* __restrict__ C, int ldc, int kslice, int vecs, int add) {
    constexpr int T = BM * BN / 64;
    __shared__ __align__(16) float As[2][SBK][BM + 4];
    __shared__ __align__(16) float Bs[2][SBK][BN + 4];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr int WN = BN / 64;                            // warps along N
    const int rm = (w / WN) * 32 + (lane >> 3) * 4, rn = (w % WN) * 64 + (lane & 7) * 4;
    const int tiles_m = (M - 1) / BM + 1;
    const int m0 = (blockIdx.x % tiles_m) * BM, n0 = (blockIdx.x / tiles_m) * BN;
    const int k0 = blockIdx.z * kslice, k1 = min(K, k0 + kslice);
    unsigned long long acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    Slab<BM, T, AKC> sa;
    Slab<BN, T, BKC> sb;
    sa.load(A, lda, m0, M, k0, k1, vecs & 1);
    sb.load(B, ldb, n0, N, k0, k1, vecs & 2);
    sa.store(As[0]);
    sb.store(Bs[0]);
    __syncthreads();
    int buf = 0;
    for (int kb = k0; kb < k1; kb += SBK, buf ^= 1) {
        const bool more = kb + SBK < k1;
        if (more) {
            sa.load(A, lda, m0, M, kb + SBK, k1, vecs & 1);
            sb.load(B, ldb, n0, N, kb + SBK, k1, vecs & 2);
        }
#pragma unroll
        for (int kk = 0; kk < SBK; ++kk) {
            float a[8];
            unsigned long long b[4];
            *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(&As[buf][kk][rm]);
            *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(&As[buf][kk][rm + 16]);
            *reinterpret_cast<ulonglong2*>(b) = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][rn]);
            *reinterpret_cast<ulonglong2*>(b + 2) = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][rn + 32]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const unsigned long long aa = pack2(a[i], a[i]);
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma2(aa, b[j], acc[i][j]);
            }
        }
        if (more) {
            sa.store(As[buf ^ 1]);
            sb.store(Bs[buf ^ 1]);
        }
        __syncthreads();
    }
    // add: 0 C = alpha acc, 1 C += alpha acc (one block per tile), 2 atomically (K split)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int gm = m0 + rm + (i < 4 ? i : 12 + i);
        if (gm >= M) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int gn = n0 + rn + 32 * h;
            float v[4];
            unpack2(acc[i][2 * h], v[0], v[1]);
            unpack2(acc[i][2 * h + 1], v[2], v[3]);
            float* c = C + (long long)gm * ldc + gn;
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] *= alpha;
            if (gn <= N - 4 && (vecs & 4)) {
                if (add == 2) {
                    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(c), "f"(v[0]), "f"(v[1]),
                                 "f"(v[2]), "f"(v[3])
                                 : "memory");
                } else {
                    float4 t = make_float4(v[0], v[1], v[2], v[3]);
                    if (add) {
                        const float4 o = *reinterpret_cast<const float4*>(c);
                        t = make_float4(o.x + t.x, o.y + t.y, o.z + t.z, o.w + t.w);
                    }
                    *reinterpret_cast<float4*>(c) = t;
                }
            } else {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (gn + q < N) {
                        if (add == 2) atomicAdd(c + q, v[q]);
                        else c[q] = add ? c[q] + v[q] : v[q];
                    }
            }
        }
    }
}

__global__ void k_scale_matrix(int M, int N, float beta, float* __restrict__ C, int ldc) {
    const long long total = (long long)M * N;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        float* c = C + (e / N) * ldc + e % N;
        *c = beta == 0.f ? 0.f : beta * *c;
    }
}

// The element-wise layers below stream their arrays once and are bound by HBM (small
// ones by the launch): four values per thread and access where the arrays allow it,
// and no 64-bit division per value.  `vec` is chosen by the launcher: 16-byte aligned
// arrays and, for the row-wise kernel, rows of a multiple of four values.

__device__ __forceinline__ float act_of(float v, int act) {
    if (act == 1) return fmaxf(v, 0.f);
    if (act == 2) return tanhf(v);
    if (act == 3) return v > 0.f ? v : 0.01f * v;
    return v;
}

// X[r][c] = act(X[r][c] + bias[c]); act: 0 none, 1 ReLU, 2 tanh, 3 Leaky ReLU (slope
// 0.01).  A block walks a chunk of columns (blockIdx.x) down its rows (blockIdx.y):
// the bias is read once per thread.  16384 x 256 tanh: 15.2 us with one value per
// thread and e % cols, 6.2 us in this form (ncu, cold).
template <int V>
__global__ void __launch_bounds__(256) k_bias_act(int rows, int cols, float* __restrict__ X,
                                                  const float* __restrict__ bias, int act) {
    const long long c = (blockIdx.x * 64LL + (threadIdx.x & 63)) * V;
    if (c >= cols) return;
    float b[V];
#pragma unroll
    for (int q = 0; q < V; ++q) b[q] = bias ? bias[c + q] : 0.f;
    for (unsigned r = blockIdx.y * 4 + (threadIdx.x >> 6); r < (unsigned)rows; r += gridDim.y * 4) {
        float* x = X + (long long)r * cols + c;
        if (V == 4) {
            float4 t = *reinterpret_cast<float4*>(x);
            t.x = act_of(t.x + b[0], act);
            t.y = act_of(t.y + b[1 % V], act);
            t.z = act_of(t.z + b[2 % V], act);
            t.w = act_of(t.w + b[3 % V], act);
            *reinterpret_cast<float4*>(x) = t;
        } else {
            x[0] = act_of(x[0] + b[0], act);
        }
    }
}

__device__ __forceinline__ float act_grad(float d, float y, int act) {
    if (act == 1) return y > 0.f ? d : 0.f;
    if (act == 2) return d * (1.f - y * y);
    if (act == 3) return y > 0.f ? d : 0.01f * d;          // the output keeps the input's sign
    return d;
}

// dX *= act'(Y), Y the activation output
__global__ void k_act_backward(long long n, float* __restrict__ dX, const float* __restrict__ Y, int act, int vec) {
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x, nth = (long long)gridDim.x * blockDim.x;
    const long long n4 = vec ? n >> 2 : 0;
    for (long long e = tid; e < n4; e += nth) {
        float4 d = reinterpret_cast<float4*>(dX)[e];
        const float4 y = reinterpret_cast<const float4*>(Y)[e];
        d.x = act_grad(d.x, y.x, act);
        d.y = act_grad(d.y, y.y, act);
        d.z = act_grad(d.z, y.z, act);
        d.w = act_grad(d.w, y.w, act);
        reinterpret_cast<float4*>(dX)[e] = d;
    }
    for (long long e = 4 * n4 + tid; e < n; e += nth) dX[e] = act_grad(dX[e], Y[e], act);
}

// db[c] = sum_r dY[r][c].  A cluster of CS blocks owns 8 columns (one 32-byte sector a
// row; narrow groups so that 256 columns still fill the chip); a warp reads 4 rows per
// load, each block takes every CS-th group of 32 rows, and rank 0 adds the blocks' sums
// from their shared memory in rank order: a fixed order, no workspace and no second
// launch.  16384 x 256: 1.4 ms with one thread per column (a single block), 9.7 us in
// this form (ncu, cold).  CS = 1 below 256 rows, where a thread adds at most 8 values.
template <int CS>
__global__ void __launch_bounds__(256) k_bias_grad(int rows, int cols, const float* __restrict__ dY,
                                                   float* __restrict__ db) {
    __shared__ float part[32][8];
    __shared__ float sums[8];
    const int tid = threadIdx.x, cc = tid & 7, rr = tid >> 3;
    const long long c = (blockIdx.x / CS) * 8LL + cc;
    const int rank = CS == 1 ? 0 : (int)(blockIdx.x % CS);
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    if (c < cols) {
        constexpr int STEP = 32 * CS;
        unsigned r = rank * 32 + rr;                       // (32 bits without the sign: r runs past rows)
        for (; r + 3 * STEP < (unsigned)rows; r += 4 * STEP)
#pragma unroll
            for (int u = 0; u < 4; ++u) s[u] += dY[(long long)(r + u * STEP) * cols + c];
        for (; r < (unsigned)rows; r += STEP) s[0] += dY[(long long)r * cols + c];
    }
    part[rr][cc] = (s[0] + s[1]) + (s[2] + s[3]);
    __syncthreads();
    if (tid < 8) {
        float t = 0.f;
        for (int q = 0; q < 32; ++q) t += part[q][tid];
        sums[tid] = t;
    }
    if (CS == 1) {
        if (tid < 8 && c < cols) db[c] = sums[tid];
        return;
    }
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    cl.sync();
    if (rank == 0 && tid < 8 && c < cols) {
        float t = 0.f;
        for (int q = 0; q < CS; ++q) t += cl.map_shared_rank(sums, q)[tid];
        db[c] = t;
    }
    cl.sync();                                             // the sums stay until rank 0 has read them
}

// The same sums, each added in the order of the rows.  BF16 training needs the bits that do
// not move with the kernel: the last bit of a bias decides BF16 roundings of the next step
// (summed in clusters, one small step in ten ended 1e-3 away from the row order).  One
// warp's issue is the bound, 4 clocks an add: a block owns 8 columns, all its threads fetch
// the next 1024 rows while 8 lanes add the current ones from shared memory, four rows a
// load: 8192 x 256 takes 30 us (40 with a load a row; 7 in clusters, in another order).
constexpr int BS_ROWS = 1024, BS_PITCH = BS_ROWS + 4;
__global__ void __launch_bounds__(256) k_bias_grad_rows(int rows, int cols, const float* __restrict__ dY,
                                                        float* __restrict__ db) {
    extern __shared__ __align__(16) float tile[];          // [2][8][BS_PITCH], column by column
    const int tid = threadIdx.x, cc = tid & 7, rr = tid >> 3;
    const long long c = blockIdx.x * 8LL + cc;
    float s = 0.f;
    // 4-byte asynchronous copies (zeros past the matrix), so that nothing waits for them here
    auto fetch = [&](unsigned r0, float* t) {
#pragma unroll 8
        for (int q = 0; q < BS_ROWS / 32; ++q) {
            const unsigned r = r0 + rr + 32 * q;
            const bool in = r < (unsigned)rows && c < cols;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                             (unsigned)__cvta_generic_to_shared(t + cc * BS_PITCH + rr + 32 * q)),
                         "l"(in ? dY + (long long)r * cols + c : dY), "r"(in ? 4 : 0)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (rows > 0) fetch(0, tile);
    int buf = 0;
    for (unsigned r0 = 0; r0 < (unsigned)rows; r0 += BS_ROWS, buf ^= 1) {
        const float* t = tile + buf * BS_PITCH * 8;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                                   // (the other buffer has been added)
        if (r0 + BS_ROWS < (unsigned)rows) fetch(r0 + BS_ROWS, tile + (buf ^ 1) * BS_PITCH * 8);
        if (tid < 8) {
            // 16 values on their way from shared memory while 16 are added; the zeros past
            // the last row leave the sum as it is
            const int m = (int)min((unsigned)BS_ROWS, (unsigned)rows - r0);
            const float4* col = reinterpret_cast<const float4*>(t + tid * BS_PITCH);
            float4 x[4], y[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = col[u];
            for (int r = 0; r < m; r += 32) {
#pragma unroll
                for (int u = 0; u < 4; ++u) y[u] = col[r / 4 + 4 + u];
#pragma unroll
                for (int u = 0; u < 4; ++u) s = (((s + x[u].x) + x[u].y) + x[u].z) + x[u].w;
                if (r + 32 < m) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) x[u] = col[r / 4 + 8 + u];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) s = (((s + y[u].x) + y[u].y) + y[u].z) + y[u].w;
            }
        }
    }
    if (tid < 8 && c < cols) db[c] = s;
}

// Adam (Kingma & Ba) with bias correction: four streams in, three out, 28 B per value.
// 134 M values: 757 us with one value per access, 561 us (6.7 TB/s, 99% of a copy) with
// four and streaming hints
__device__ __forceinline__ void adam_one(float& p, float g, float& m, float& v, float lr, float b1, float b2, float eps,
                                         float c1, float c2) {
    // (the fused multiply-adds spelled out, so that vector and scalar paths give the same bits)
    m = fmaf(1.f - b1, g, __fmul_rn(b1, m));
    v = fmaf(__fmul_rn(1.f - b2, g), g, __fmul_rn(b2, v));
    p -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

__global__ void __launch_bounds__(256) k_adam(long long n, float* __restrict__ p, const float* __restrict__ g,
                                              float* __restrict__ m, float* __restrict__ v, float lr, float b1,
                                              float b2, float eps, float c1, float c2, int vec) {
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x, nth = (long long)gridDim.x * blockDim.x;
    const long long n4 = vec ? n >> 2 : 0;
    for (long long e = tid; e < n4; e += nth) {
        const float4 g4 = __ldcs(reinterpret_cast<const float4*>(g) + e);
        float4 m4 = __ldcs(reinterpret_cast<float4*>(m) + e), v4 = __ldcs(reinterpret_cast<float4*>(v) + e);
        float4 p4 = __ldcs(reinterpret_cast<float4*>(p) + e);
        adam_one(p4.x, g4.x, m4.x, v4.x, lr, b1, b2, eps, c1, c2);
        adam_one(p4.y, g4.y, m4.y, v4.y, lr, b1, b2, eps, c1, c2);
        adam_one(p4.z, g4.z, m4.z, v4.z, lr, b1, b2, eps, c1, c2);
        adam_one(p4.w, g4.w, m4.w, v4.w, lr, b1, b2, eps, c1, c2);
        __stcs(reinterpret_cast<float4*>(m) + e, m4);
        __stcs(reinterpret_cast<float4*>(v) + e, v4);
        __stcs(reinterpret_cast<float4*>(p) + e, p4);
    }
    for (long long e = 4 * n4 + tid; e < n; e += nth) {
        float pe = p[e], me = m[e], ve = v[e];
        adam_one(pe, g[e], me, ve, lr, b1, b2, eps, c1, c2);
        m[e] = me;
        v[e] = ve;
        p[e] = pe;
    }
}

// Relative-L2 loss of the DeepONet output on sampled nodes.
// pred, target: B x (2P) with the real parts in columns [0, P) and the imaginary
// parts in [P, 2P).  loss[b] = ||pred_b - target_b||^2 / ||target_b||^2;
// dpred = d(mean_b loss[b]) / d pred.  A cluster of CS blocks per sample: rank 0 takes
// the two sums (thread t adds entries t, t + 256, ... in order; its loads do not depend
// on the chain of adds, so 16 of each array are in flight), every block reads them from
// rank 0's shared memory and scales its own share.  The order of the sums is that of one
// block per sample, because in BF16 training the last bit of dpred decides roundings
// further down.  32 x 32768: 86.6 us as one block per sample with one load
// in flight per chain, 16.0 us in this form (ncu, cold).
template <int CS>
__global__ void __launch_bounds__(256) k_rel_l2(int Bn, int P2, const float* __restrict__ pred,
                                                const float* __restrict__ target, float* __restrict__ dpred,
                                                float* __restrict__ loss) {
    __shared__ float s_num[8], s_den[8];
    __shared__ float sums[2];
    const int b = blockIdx.x / CS, rank = CS == 1 ? 0 : (int)(blockIdx.x % CS);
    const float* pr = pred + (long long)b * P2;
    const float* tg = target + (long long)b * P2;
    float a = 0.f, c = 0.f;
    if (rank == 0) {
        float num = 0.f, den = 0.f;
#pragma unroll 16
        for (unsigned e = threadIdx.x; e < (unsigned)P2; e += 256) {
            const float t = tg[e], d = pr[e] - t;
            num = fmaf(d, d, num);
            den = fmaf(t, t, den);
        }
        for (int o = 16; o > 0; o >>= 1) {
            num += __shfl_xor_sync(0xffffffffu, num, o);
            den += __shfl_xor_sync(0xffffffffu, den, o);
        }
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        if (lane == 0) { s_num[w] = num; s_den[w] = den; }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 0; q < 8; ++q) { a += s_num[q]; c += s_den[q]; }
            sums[0] = a;
            sums[1] = c;
            loss[b] = a / c;
        }
    }
    if (CS == 1) {
        __syncthreads();
        c = sums[1];
    } else {
        cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
        cl.sync();
        c = cl.map_shared_rank(sums, 0)[1];
        cl.sync();                                         // the sums stay until every block has read them
    }
    const unsigned share = ((unsigned)P2 + CS - 1) / CS, e0 = min((unsigned)P2, rank * share);
    const unsigned e1 = min((unsigned)P2, e0 + share);
    const float scale = 2.f / (c * Bn);
#pragma unroll 4
    for (unsigned e = e0 + threadIdx.x; e < e1; e += 256) dpred[(long long)b * P2 + e] = scale * (pr[e] - tg[e]);
}

// dst[r][c] = src[ri[r]][ci[c]] (ri, ci may be null: identity)
__global__ void k_gather(int rows, int cols, const float* __restrict__ src, long long lds, const int* __restrict__ ri,
                         const int* __restrict__ ci, float* __restrict__ dst) {
    const long long total = (long long)rows * cols;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int r = (int)(e / cols), c = (int)(e % cols);
        const long long sr = ri ? ri[r] : r;
        const long long sc = ci ? ci[c] : c;
        dst[e] = src[sr * lds + sc];
    }
}

int grid_for(long long n) {
    long long b = (n + 255) / 256;
    return (int)(b < 8 * 152 ? (b < 1 ? 1 : b) : 8 * 152);
}

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// a launch of `blocks` blocks in clusters of CS (CS divides blocks)
template <typename... KArgs, typename... Args>
cudaError_t launch_clustered(void (*kern)(KArgs...), unsigned blocks, unsigned cs, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cs;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// ---- 3D convolution of the CNN branch (App. B): 3 x 3 x 3 kernels, stride s, zero
// padding pad, layout [batch][channel][z][y][x], W[out][in][kz][ky][kx].  Every output
// value is summed by one thread (inputs, then kz, ky, kx) or one block (fixed tree),
// so the results do not depend on scheduling.
constexpr int CK = 3;

__device__ __forceinline__ long long vox(int D, int z, int y, int x) { return ((long long)z * D + y) * D + x; }

// Y[b][o][.] = bias[o] + sum_{i,k} W[o][i][k] X[b][i][. s + k - pad]
__global__ void k_conv3d(int B, int Ci, int D, int Co, int Do, int stride, int pad, const float* __restrict__ X,
                         const float* __restrict__ W, const float* __restrict__ bias, float* __restrict__ Y) {
    const long long V = (long long)Do * Do * Do, total = (long long)B * Co * V;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const long long v = e % V;
        const int o = (int)((e / V) % Co), b = (int)(e / (V * Co));
        const int ox = (int)(v % Do), oy = (int)((v / Do) % Do), oz = (int)(v / ((long long)Do * Do));
        float acc = 0.f;
        for (int i = 0; i < Ci; ++i) {
            const float* xi = X + ((long long)b * Ci + i) * D * D * D;
            const float* wi = W + ((long long)o * Ci + i) * CK * CK * CK;
            for (int kz = 0; kz < CK; ++kz) {
                const int z = oz * stride + kz - pad;
                if (z < 0 || z >= D) continue;
                for (int ky = 0; ky < CK; ++ky) {
                    const int y = oy * stride + ky - pad;
                    if (y < 0 || y >= D) continue;
                    for (int kx = 0; kx < CK; ++kx) {
                        const int x = ox * stride + kx - pad;
                        if (x < 0 || x >= D) continue;
                        acc = fmaf(wi[(kz * CK + ky) * CK + kx], xi[vox(D, z, y, x)], acc);
                    }
                }
            }
        }
        Y[e] = acc + (bias ? bias[o] : 0.f);
    }
}

// dX[b][i][p] = sum_{o,k} W[o][i][k] dY[b][o][q] over the outputs q that read p with offset k
__global__ void k_conv3d_dx(int B, int Ci, int D, int Co, int Do, int stride, int pad, const float* __restrict__ W,
                            const float* __restrict__ dY, float* __restrict__ dX) {
    const long long V = (long long)D * D * D, total = (long long)B * Ci * V, Vo = (long long)Do * Do * Do;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const long long v = e % V;
        const int i = (int)((e / V) % Ci), b = (int)(e / (V * Ci));
        const int x = (int)(v % D), y = (int)((v / D) % D), z = (int)(v / ((long long)D * D));
        float acc = 0.f;
        for (int o = 0; o < Co; ++o) {
            const float* dyo = dY + ((long long)b * Co + o) * Vo;
            const float* wo = W + ((long long)o * Ci + i) * CK * CK * CK;
            for (int kz = 0; kz < CK; ++kz) {
                const int tz = z + pad - kz;
                if (tz < 0 || tz % stride) continue;
                const int oz = tz / stride;
                if (oz >= Do) continue;
                for (int ky = 0; ky < CK; ++ky) {
                    const int ty = y + pad - ky;
                    if (ty < 0 || ty % stride) continue;
                    const int oy = ty / stride;
                    if (oy >= Do) continue;
                    for (int kx = 0; kx < CK; ++kx) {
                        const int tx = x + pad - kx;
                        if (tx < 0 || tx % stride) continue;
                        const int ox = tx / stride;
                        if (ox >= Do) continue;
                        acc = fmaf(wo[(kz * CK + ky) * CK + kx], dyo[vox(Do, oz, oy, ox)], acc);
                    }
                }
            }
        }
        dX[e] = acc;
    }
}

// one block per weight (o, i, k) (and per bias o when i == Ci): the sum over the batch
// and the outputs of dY X at the offset, in a fixed order (strided per thread, then a
// shared-memory tree)
__global__ void __launch_bounds__(256) k_conv3d_dw(int B, int Ci, int D, int Co, int Do, int stride, int pad,
                                                   const float* __restrict__ X, const float* __restrict__ dY,
                                                   float* __restrict__ dW, float* __restrict__ db) {
    __shared__ float red[256];
    const int wid = blockIdx.x;                          // o * (Ci * 27 + 1) + i * 27 + k, k = 27: bias
    const int per = Ci * CK * CK * CK + 1;
    const int o = wid / per, r = wid % per;
    const bool is_bias = r == per - 1;
    const int i = is_bias ? 0 : r / (CK * CK * CK), k = is_bias ? 0 : r % (CK * CK * CK);
    const int kz = k / (CK * CK), ky = (k / CK) % CK, kx = k % CK;
    const long long Vo = (long long)Do * Do * Do, total = (long long)B * Vo;
    float acc = 0.f;
    for (long long e = threadIdx.x; e < total; e += blockDim.x) {
        const int b = (int)(e / Vo);
        const long long v = e % Vo;
        const float g = dY[((long long)b * Co + o) * Vo + v];
        if (is_bias) {
            acc += g;
            continue;
        }
        const int ox = (int)(v % Do), oy = (int)((v / Do) % Do), oz = (int)(v / ((long long)Do * Do));
        const int z = oz * stride + kz - pad, y = oy * stride + ky - pad, x = ox * stride + kx - pad;
        if (z < 0 || z >= D || y < 0 || y >= D || x < 0 || x >= D) continue;
        acc = fmaf(g, X[((long long)b * Ci + i) * D * D * D + vox(D, z, y, x)], acc);
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (is_bias) {
            if (db) db[o] = red[0];
        } else if (dW) {
            dW[((long long)o * Ci + i) * CK * CK * CK + k] = red[0];
        }
    }
}

}  // namespace

extern "C" {

helm_status nn_gemm(int transA, int transB, int M, int N, int K, float alpha, const float* A, int lda, const float* B,
                    int ldb, float beta, float* C, int ldc, void* stream) {
    if (M < 0 || N < 0 || K < 0 || !C || (K > 0 && (!A || !B))) return HELM_BAD_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (M == 0 || N == 0) return HELM_OK;
    if (K == 0 || alpha == 0.f) {
        if (beta != 1.f) k_scale_matrix<<<grid_for((long long)M * N), 256, 0, s>>>(M, N, beta, C, ldc);
        return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
    }
    // K is split, and the parts added atomically in any order, only where K is long and C
    // small: from 128 on and below 304 tiles of 64 x 64.  Other products are one chain a
    // value, the same bits on every call
    const auto up = [](long long a, long long b) { return (a + b - 1) / b; };
    const bool split = K >= 128 && up(M, 64) * up(N, 64) < 2 * 152;
    // 128 x 128 tiles where M fills them; 32 rows for the batch-sized products (a row of
    // the batch per 8 threads wastes nothing on padding), and for an unsplit product of few
    // tiles: one 32 x 256 tile an SM (4864 x 256 x 256: 30.8 -> 22.6 us; with 188 of them
    // 30.8 -> 32.9) or two 32 x 128 (9728 x 100 x 100: 16.4 -> 12.4).  256 columns for N > 128
    const int wide = N > 128 ? 256 : 128;
    const int bm = M <= 64 || (!split && up(M, 32) * up(N, wide) <= (wide == 256 ? 152 : 2 * 152)) ? 32 : 128;
    const int bn = bm == 32 ? wide : 128;
    const long long tiles = up(M, bm) * up(N, bn);
    if (tiles > 0x7fffffffLL) return HELM_BAD_ARG;
    // a split fills every SM's resident blocks once (2 of 256 threads, 3 of 128, 5 of 64: a
    // part of a second wave would cost a whole one), at least 2 slabs each
    const long long want = (bm == 128 ? 2 : bn == 256 ? 3 : 5) * 152;
    int splits = split ? (int)std::max<long long>(1, std::min<long long>(want / tiles, K / (2 * SBK))) : 1;
    int kslice = ((K + splits - 1) / splits + SBK - 1) / SBK * SBK;
    splits = (K + kslice - 1) / kslice;
    int add = splits > 1 ? 2 : (beta != 0.f);
    if (beta != 1.f && add) {
        if (beta == 0.f && (M == 1 || ldc == N)) {
            if (cudaMemsetAsync(C, 0, sizeof(float) * N * (size_t)M, s) != cudaSuccess) return HELM_CUDA_ERROR;
        } else if (beta == 0.f && ldc > N) {
            if (cudaMemset2DAsync(C, sizeof(float) * ldc, 0, sizeof(float) * N, M, s) != cudaSuccess)
                return HELM_CUDA_ERROR;
        } else {
            k_scale_matrix<<<grid_for((long long)M * N), 256, 0, s>>>(M, N, beta, C, ldc);
        }
    }
    const int vecs = (lda % 4 == 0 && al16(A) ? 1 : 0) | (ldb % 4 == 0 && al16(B) ? 2 : 0) |
                     (ldc % 4 == 0 && al16(C) ? 4 : 0);
    const dim3 g((unsigned)tiles, 1, (unsigned)splits);
#define SG(BM, BN, AKC, BKC)                                                                                   \
    k_sgemm<BM, BN, AKC, BKC><<<g, BM * BN / 64, 0, s>>>(M, N, K, alpha, A, lda, B, ldb, C, ldc, kslice, vecs, add)
#define SGT(BM, BN)                                                      \
    do {                                                                 \
        if (!transA && transB) SG(BM, BN, true, true);                   \
        else if (!transA) SG(BM, BN, true, false);                       \
        else if (transB) SG(BM, BN, false, true);                        \
        else SG(BM, BN, false, false);                                   \
    } while (0)
    if (bm == 128) SGT(128, 128);
    else if (bn == 256) SGT(32, 256);
    else SGT(32, 128);
#undef SGT
#undef SG
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

helm_status nn_bias_act(int rows, int cols, float* X, const float* bias, int act, void* stream) {
    if (rows < 0 || cols < 0 || !X || act < 0 || act > 3) return HELM_BAD_ARG;
    if (rows == 0 || cols == 0) return HELM_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool vec = cols % 4 == 0 && al16(X);
    const int gx = (cols - 1) / (vec ? 256 : 64) + 1;
    const dim3 g(gx, (unsigned)std::max(1, std::min((rows - 1) / 4 + 1, 8 * 152 / std::min(gx, 8 * 152))));
    if (vec) k_bias_act<4><<<g, 256, 0, s>>>(rows, cols, X, bias, act);
    else k_bias_act<1><<<g, 256, 0, s>>>(rows, cols, X, bias, act);
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

helm_status nn_act_backward(long long n, float* dX, const float* Y, int act, void* stream) {
    if (n < 0 || !dX || !Y || act < 0 || act > 3) return HELM_BAD_ARG;
    const int vec = al16(dX) && al16(Y);
    k_act_backward<<<grid_for(vec ? (n + 3) / 4 : n), 256, 0, static_cast<cudaStream_t>(stream)>>>(n, dX, Y, act, vec);
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

helm_status nn_bias_grad(int rows, int cols, const float* dY, float* db, void* stream) {
    if (rows < 0 || cols < 0 || !dY || !db) return HELM_BAD_ARG;
    if (cols == 0) return HELM_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const unsigned groups = (unsigned)((cols - 1) / 8 + 1);
    if (rows < 256) k_bias_grad<1><<<groups, 256, 0, s>>>(rows, cols, dY, db);
    else if (launch_clustered(k_bias_grad<8>, 8 * groups, 8, s, rows, cols, dY, db) != cudaSuccess) return HELM_CUDA_ERROR;
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

helm_status nn_bias_grad_rows(int rows, int cols, const float* dY, float* db, void* stream) {
    if (rows < 0 || cols < 0 || !dY || !db) return HELM_BAD_ARG;
    if (cols == 0) return HELM_OK;
    const size_t smem = 2 * BS_PITCH * 8 * sizeof(float);
    if (cudaFuncSetAttribute(k_bias_grad_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return HELM_CUDA_ERROR;
    k_bias_grad_rows<<<(cols - 1) / 8 + 1, 256, smem, static_cast<cudaStream_t>(stream)>>>(rows, cols, dY, db);
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

helm_status nn_adam(long long n, float* p, const float* g, float* m, float* v, float lr, float beta1, float beta2,
                    float eps, int t, void* stream) {
    if (n < 0 || !p || !g || !m || !v || t < 1) return HELM_BAD_ARG;
    const float c1 = 1.f - powf(beta1, (float)t), c2 = 1.f - powf(beta2, (float)t);
    const int vec = al16(p) && al16(g) && al16(m) && al16(v);
    k_adam<<<grid_for(vec ? (n + 3) / 4 : n), 256, 0, static_cast<cudaStream_t>(stream)>>>(n, p, g, m, v, lr, beta1,
                                                                                         beta2, eps, c1, c2, vec);
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

helm_status nn_gather(int rows, int cols, const float* src, long long lds, const int* row_idx, const int* col_idx,
                      float* dst, void* stream) {
    if (rows < 0 || cols < 0 || !src || !dst) return HELM_BAD_ARG;
    k_gather<<<grid_for((long long)rows * cols), 256, 0, static_cast<cudaStream_t>(stream)>>>(rows, cols, src, lds, row_idx,
                                                                                             col_idx, dst);
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

helm_status nn_rel_l2(int B, int P2, const float* pred, const float* target, float* dpred, float* loss, void* stream) {
    if (B < 1 || P2 < 1 || !pred || !target || !dpred || !loss) return HELM_BAD_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // (a block alone writes up to 16 values per thread before a cluster pays for its barriers)
    if (P2 <= 4096 || (long long)B * 4 > 0x7fffffffLL) k_rel_l2<1><<<B, 256, 0, s>>>(B, P2, pred, target, dpred, loss);
    else if (launch_clustered(k_rel_l2<4>, 4u * (unsigned)B, 4, s, B, P2, pred, target, dpred, loss) != cudaSuccess)
        return HELM_CUDA_ERROR;
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

helm_status nn_conv3d(int B, int Ci, int D, int Co, int stride, int pad, const float* X, const float* W,
                      const float* bias, float* Y, void* stream) {
    if (B < 1 || Ci < 1 || Co < 1 || D < 1 || stride < 1 || pad < 0 || pad > 2 || !X || !W || !Y) return HELM_BAD_ARG;
    const int Do = (D + 2 * pad - CK) / stride + 1;
    if (D + 2 * pad < CK || Do < 1) return HELM_BAD_ARG;
    k_conv3d<<<grid_for((long long)B * Co * Do * Do * Do), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        B, Ci, D, Co, Do, stride, pad, X, W, bias, Y);
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

helm_status nn_conv3d_backward(int B, int Ci, int D, int Co, int stride, int pad, const float* X, const float* W,
                               const float* dY, float* dX, float* dW, float* db, void* stream) {
    if (B < 1 || Ci < 1 || Co < 1 || D < 1 || stride < 1 || pad < 0 || pad > 2 || !dY) return HELM_BAD_ARG;
    if ((dX && !W) || ((dW || db) && !X)) return HELM_BAD_ARG;
    const int Do = (D + 2 * pad - CK) / stride + 1;
    if (D + 2 * pad < CK || Do < 1) return HELM_BAD_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (dX)
        k_conv3d_dx<<<grid_for((long long)B * Ci * D * D * D), 256, 0, s>>>(B, Ci, D, Co, Do, stride, pad, W, dY, dX);
    if (dW || db)
        k_conv3d_dw<<<Co * (Ci * CK * CK * CK + 1), 256, 0, s>>>(B, Ci, D, Co, Do, stride, pad, X, dY, dW, db);
    return cudaGetLastError() == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

}  // extern "C"
