// BF16 GEMM with FP32 accumulation on the fifth-generation tensor cores (tcgen05),
// for the dense layers of the DeepONet (App. B): C = alpha op(A) op(B) + beta C with
// FP32 row-major operands, as nn_gemm, but with op(A) and op(B) rounded to BF16.
//
// Structure:
//  - both operands are first converted to BF16 "K-major" copies (op(B)^T as N x K rows,
//    op(A) as M x K rows) in one launch, zero-padded to multiples of 128 rows and 64
//    columns so that every TMA box lies inside the copy and starts on a 16-byte boundary;
//  - a CTA owns 128 columns of C (the M = 128 side of the MMA, so that the 32 lanes of an
//    epilogue warp hold neighbouring columns and its stores coalesce) and TN rows of C (the
//    N side): 16 to 128, as few as leave about one CTA per SM.  K is not split: the sum of
//    each value stays one chain, whatever the tile;
//  - warp 0: one elected thread loads the two boxes of every 64-deep K step with
//    cp.async.bulk.tensor (128-byte swizzle); a stage is SUB such steps on one "full"
//    mbarrier, and the ring has as many stages as K fills, up to the three that 222 KB hold;
//  - warp 1: one elected thread issues tcgen05.mma.kind::f16 (K = 16 per instruction, four
//    per step) into a TMEM accumulator and commits each stage to its "empty" mbarrier, the
//    last one to the "done" mbarrier as well;
//  - warp 2 allocates and frees the TMEM columns;
//  - warps 4-7 (one per quarter of the TMEM lanes) read the accumulator with
//    tcgen05.ld and write alpha D + beta C for the valid rows and columns.
// What bounds it: the branch's first layer (64 x 256 x 128000 at 40^3) is a chain of 8000
// dependent MMAs per value on 8 CTAs.  An MMA takes about 27 ns whatever its width, and one
// round of wait and commit about 150 ns of the issuing thread (measured with the loads, the
// MMAs and the commits left out in turn), so a stage holds as many K steps as still leave
// three stages: per step 330 ns with one step a stage and a lane == 0 branch, 251 elected,
// 178 with two steps, 146 with three, 131 with four (145 with six, which leaves two stages).
// Looking at the next stage's barrier before the MMAs gains with one or two steps and loses
// with more.  64 x 256 x 128000: 660 -> 262 us.  Splitting K would shorten it further but
// change the last bits of the activations, which the next layer rounds to BF16.  The weight
// gradient (K = 64, 256 x 128000 values) is bound by the stores: 32 us.
// Every mbarrier wait is bounded: a wait that runs out records an error flag and the
// thread goes on (the result is then garbage but the launch ends); the host reads
// the flag with nn_gemm_bf16_status.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "helm_internal.cuh"

namespace helm {

namespace {

constexpr int TBM = 128, TBK = 64, MAX_STAGES = 3;       // (three stages of every tile fill the ring)
constexpr int TC_THREADS = 256;
constexpr unsigned kRingBytes = 222 * 1024;                    // shared memory of the stages, at most
constexpr unsigned kWaitLimit = 1u << 26;

__device__ int g_tc_error;

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, unsigned parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(su32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait for the phase of the given parity; false (and the error flag) on a timeout.
// Once a wait of the launch has given up the others do so too, at their next look at the
// flag.  They look only while waiting in vain: the flag lies in global memory, and a look
// before every wait cost the MMA thread 0.4 us per K step (0.46 us a step whatever the
// tile or the number of stages).
__device__ __forceinline__ bool mbar_wait(uint64_t* b, unsigned parity) {
    for (unsigned it = 1; it <= kWaitLimit; ++it) {
        if (mbar_try(b, parity)) return true;
        if ((it & 1023u) == 0 && *reinterpret_cast<volatile int*>(&g_tc_error)) return false;
    }
    atomicExch(&g_tc_error, 1);
    return false;
}

// true in one lane of the warp (all lanes arrive).  The issuing instructions take their
// operands from uniform registers; inside a lane == 0 branch the compiler moves every one
// there through a loop over the lanes.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(su32(dst)), "l"(map), "r"(x), "r"(y), "r"(su32(bar))
        : "memory");
}

// shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups
// 1024 bytes apart (start address and offsets in units of 16 bytes)
__device__ __forceinline__ uint64_t smem_desc(const void* p) {
    const uint64_t addr = (su32(p) & 0x3FFFFu) >> 4;
    return addr | (uint64_t(1) << 16) | (uint64_t(1024 >> 4) << 32) | (uint64_t(1) << 46) | (uint64_t(2) << 61);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// C (M x N) = alpha A B^T + beta C from the K-major copies; mapN: op(B)^T, mapM: op(A)
template <int TN, int SUB>
__global__ void __launch_bounds__(TC_THREADS)
    k_gemm_bf16_tc(const __grid_constant__ CUtensorMap mapN, const __grid_constant__ CUtensorMap mapM, int M, int N,
                   int Kp, int stages, float alpha, float beta, float* __restrict__ C, int ldc) {
    constexpr unsigned kNBytes = TBM * TBK * 2, kMBytes = TN * TBK * 2;
    constexpr unsigned kCols = TN < 32 ? 32 : TN;          // TMEM columns (at least 32 are allocated)
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // 1024-byte alignment of the stage buffers (the swizzle atom)
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sN = smem;
    uint8_t* sM = smem + min(stages * SUB, Kp / TBK) * kNBytes;
    __shared__ uint64_t full[MAX_STAGES], empty[MAX_STAGES], done;
    __shared__ uint32_t tmem_base;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles_m = (M + TN - 1) / TN;
    const int m0 = (blockIdx.x % tiles_m) * TN, n0 = (blockIdx.x / tiles_m) * TBM;
    const int nk = Kp / TBK;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tmem_base)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;

    if (warp == 0) {
        // producer
        int s = 0;
        unsigned parity = 1;                               // (the first round finds every stage empty)
        for (int kb = 0, g = 0; kb < nk; kb += SUB, ++g) {
            if (g >= stages) mbar_wait(&empty[s], parity);
            if (elect_one()) {
                const int sub = min(SUB, nk - kb);
                mbar_expect_tx(&full[s], sub * (kNBytes + kMBytes));
#pragma unroll
                for (int u = 0; u < SUB; ++u)
                    if (u < sub) {
                        tma_load_2d(sN + (s * SUB + u) * kNBytes, &mapN, (kb + u) * TBK, n0, &full[s]);
                        tma_load_2d(sM + (s * SUB + u) * kMBytes, &mapM, (kb + u) * TBK, m0, &full[s]);
                    }
            }
            if (++s == stages) {
                s = 0;
                parity ^= 1u;
            }
        }
    } else if (warp == 1) {
        // MMA issuer
        constexpr uint32_t idesc = idesc_bf16(TBM, TN);
        const uint64_t dn0 = smem_desc(sN), dm0 = smem_desc(sM);
        int s = 0;
        unsigned parity = 0;
        for (int kb = 0; kb < nk; kb += SUB) {
            mbar_wait(&full[s], parity);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (elect_one()) {
#pragma unroll
                for (int u = 0; u < SUB; ++u) {
                    if (kb + u < nk) {
                        const uint64_t da = dn0 + (uint64_t)((s * SUB + u) * (kNBytes >> 4));
                        const uint64_t db = dm0 + (uint64_t)((s * SUB + u) * (kMBytes >> 4));
#pragma unroll
                        for (int k = 0; k < TBK / 16; ++k) {
                            // K = 16 BF16 = 32 bytes further along the swizzled 128-byte rows
                            const uint64_t koff = (uint64_t)((k * 32) >> 4);
                            const uint32_t acc = (kb > 0 || u > 0 || k > 0) ? 1u : 0u;
                            asm volatile(
                                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                                " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                                "l"(da + koff), "l"(db + koff), "r"(idesc), "r"(acc)
                                : "memory");
                        }
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 su32(&empty[s]))
                             : "memory");
                if (kb + SUB >= nk)
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                     su32(&done))
                                 : "memory");
            }
            if (++s == stages) {
                s = 0;
                parity ^= 1u;
            }
        }
    } else if (warp >= 4) {
        // epilogue: warp 4 + q reads TMEM lanes 32 q .. 32 q + 31 (columns n of the tile)
        const int q = warp - 4;
        mbar_wait(&done, 0);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int n = n0 + 32 * q + lane;
        for (int c0 = 0; c0 < TN; c0 += 16) {
            uint32_t v[16];
            const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c0;
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                "%14, %15}, [%16];"
                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                  "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                : "r"(taddr)
                : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (n < N) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int m = m0 + c0 + j;
                    if (m < M) {
                        float* c = C + (long long)m * ldc + n;
                        const float d = __uint_as_float(v[j]);
                        *c = beta == 0.f ? alpha * d : fmaf(alpha, d, beta * *c);
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 2) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
    }
}

// one operand to convert: dst (rows_p x Kp, BF16, row-major, zero padding); element (r, k)
// is X[r * ld + k] (kc) or X[k * ld + r]; vec: 16-byte rows and base
struct PackOp {
    const float* X;
    __nv_bfloat16* dst;
    int ld, rows, rows_p, kc, vec;
};

__device__ __forceinline__ uint4 bf16x8_of(const float* v) {
    uint4 u;
    __nv_bfloat162 p[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) p[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
    u.x = *reinterpret_cast<const uint32_t*>(&p[0]);
    u.y = *reinterpret_cast<const uint32_t*>(&p[1]);
    u.z = *reinterpret_cast<const uint32_t*>(&p[2]);
    u.w = *reinterpret_cast<const uint32_t*>(&p[3]);
    return u;
}

// four values along the contiguous side, zeros past n
__device__ __forceinline__ float4 load4(const float* p, int n, bool vec) {
    if (n >= 4 && vec) return __ldg(reinterpret_cast<const float4*>(p));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n > 0) v.x = __ldg(p);
    if (n > 1) v.y = __ldg(p + 1);
    if (n > 2) v.z = __ldg(p + 2);
    if (n > 3) v.w = __ldg(p + 3);
    return v;
}

// Both operands to K-major BF16, 64 rows x 64 k a block, 16 bytes per load and store: the
// copies stream at HBM's rate.  An operand stored with its rows contiguous goes through
// shared memory.  22 launches of a training step at 40^3 take about 180 us; as 44 launches
// with one element per thread, a 64-bit division each and reads a whole row apart, 476 us.
__global__ void __launch_bounds__(256) k_pack_bf16(PackOp a, PackOp b, int K, int Kp, long long blocks_a) {
    __shared__ float tile[64][65];
    const bool second = blockIdx.x >= blocks_a;
    const PackOp o = second ? b : a;
    const long long blk = blockIdx.x - (second ? blocks_a : 0);
    const int kt = Kp / TBK;
    const int r0 = (int)(blk / kt) * 64, k0 = (int)(blk % kt) * TBK, t = threadIdx.x;
    const int c = t & 7;                                   // chunk of eight k of the rows t / 8, t / 8 + 32
    float v[2][8];
    if (o.kc) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int r = r0 + (t >> 3) + 32 * u, k = k0 + 8 * c;
            const int n = r < o.rows ? K - k : 0;
            const float* p = o.X + (long long)r * o.ld + k;
            const float4 x = load4(p, n, o.vec), y = load4(p + 4, n - 4, o.vec);
            v[u][0] = x.x; v[u][1] = x.y; v[u][2] = x.z; v[u][3] = x.w;
            v[u][4] = y.x; v[u][5] = y.y; v[u][6] = y.z; v[u][7] = y.w;
        }
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = (t >> 4) + 16 * u, r = 4 * (t & 15);
            const int n = k0 + k < K ? o.rows - (r0 + r) : 0;
            const float4 x = load4(o.X + (long long)(k0 + k) * o.ld + r0 + r, n, o.vec);
            tile[r][k] = x.x;
            tile[r + 1][k] = x.y;
            tile[r + 2][k] = x.z;
            tile[r + 3][k] = x.w;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int q = 0; q < 8; ++q) v[u][q] = tile[(t >> 3) + 32 * u][8 * c + q];
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int r = r0 + (t >> 3) + 32 * u;
        if (r < o.rows_p) *reinterpret_cast<uint4*>(o.dst + (long long)r * Kp + k0 + 8 * c) = bf16x8_of(v[u]);
    }
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
    static EncodeFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, []() {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeFn>(p);
    });
    return fn;
}

bool make_map(CUtensorMap* map, const void* base, int rows_p, int Kp, int box_rows) {
    EncodeFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)Kp, (cuuint64_t)rows_p};
    const cuuint64_t strides[1] = {(cuuint64_t)Kp * 2};
    const cuuint32_t box[2] = {TBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// per-device workspace of the BF16 copies (grown on demand, held until exit).  Each call
// first waits for the last one's event, so that calls on different streams take turns (not
// while being captured: a captured call is ordered by its graph)
struct Ws {
    void* p = nullptr;
    size_t bytes = 0;
    cudaEvent_t ev = nullptr;
    bool used = false;
};
std::mutex g_ws_mutex;
Ws g_ws[64];

template <int TN, int SUB>
cudaError_t gemm_tc(const CUtensorMap& mn, const CUtensorMap& mm, int M, int N, int Kp, float alpha, float beta, float* C,
                    int ldc, cudaStream_t s) {
    constexpr unsigned stage = (TBM + TN) * TBK * 2 * SUB;
    static_assert(MAX_STAGES * stage <= kRingBytes && (MAX_STAGES + 1) * stage > kRingBytes, "the ring holds MAX_STAGES");
    const int stages = std::min((Kp / TBK + SUB - 1) / SUB, MAX_STAGES);
    const size_t smem = (size_t)std::min(stages * SUB, Kp / TBK) * (stage / SUB) + 1024;
    const cudaError_t e =
        cudaFuncSetAttribute(k_gemm_bf16_tc<TN, SUB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kRingBytes + 1024));
    if (e != cudaSuccess) return e;
    const long long tiles = (long long)((M + TN - 1) / TN) * ((N + TBM - 1) / TBM);
    k_gemm_bf16_tc<TN, SUB><<<(unsigned)tiles, TC_THREADS, smem, s>>>(mn, mm, M, N, Kp, stages, alpha, beta, C, ldc);
    return cudaGetLastError();
}

}  // namespace

}  // namespace helm

using namespace helm;

extern "C" helm_status nn_gemm_bf16(int transA, int transB, int M, int N, int K, float alpha, const float* A, int lda,
                                    const float* B, int ldb, float beta, float* C, int ldc, void* stream) {
    if (M < 0 || N < 0 || K < 0 || !A || !B || !C || ldc < N) return HELM_BAD_ARG;
    if (M == 0 || N == 0) return HELM_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int Mp = (M + TBM - 1) / TBM * TBM, Np = (N + TBM - 1) / TBM * TBM;
    const int Kp = K == 0 ? TBK : (K + TBK - 1) / TBK * TBK;
    const size_t need = ((size_t)Mp + Np) * Kp * 2;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return HELM_NO_DEVICE;
    std::lock_guard<std::mutex> lock(g_ws_mutex);
    Ws& w = g_ws[dev];
    if (w.bytes < need) {
        if (w.p) {
            cudaStreamSynchronize(s);
            cudaFree(w.p);
        }
        w.p = nullptr;
        w.bytes = 0;
        if (cudaMalloc(&w.p, need) != cudaSuccess) {
            cudaGetLastError();
            return HELM_OUT_OF_MEMORY;
        }
        w.bytes = need;
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) return HELM_CUDA_ERROR;
    const bool ordered = cap == cudaStreamCaptureStatusNone;
    if (!w.ev && cudaEventCreateWithFlags(&w.ev, cudaEventDisableTiming) != cudaSuccess) return HELM_CUDA_ERROR;
    if (ordered && w.used && cudaStreamWaitEvent(s, w.ev, 0) != cudaSuccess) return HELM_CUDA_ERROR;
    __nv_bfloat16* Ab = static_cast<__nv_bfloat16*>(w.p);
    __nv_bfloat16* Bb = Ab + (size_t)Mp * Kp;
    auto vec = [](const float* p, int ld) { return ld % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    // op(B) is K x N; its K-major copy holds op(B)^T (N x K): element (n, k) = op(B)(k, n)
    const PackOp pa{A, Ab, lda, M, Mp, !transA, vec(A, lda)}, pb{B, Bb, ldb, N, Np, transB != 0, vec(B, ldb)};
    const long long ka = (long long)(Mp / 64) * (Kp / TBK), kb = (long long)(Np / 64) * (Kp / TBK);
    if (ka + kb > 0x7fffffffLL) return HELM_BAD_ARG;
    k_pack_bf16<<<(unsigned)(ka + kb), 256, 0, s>>>(pa, pb, K, Kp, ka);
    // the tallest tile (fewest reads of op(B)) that still gives about one CTA per SM
    const long long nt = Np / TBM;
    int tn = 128;
    while (tn > 16 && nt * ((M + tn - 1) / tn) < 128) tn /= 2;
    while (tn > 16 && tn / 2 >= M) tn /= 2;                // (no taller than the rows there are)
    CUtensorMap mn, mm;
    if (!make_map(&mn, Bb, Np, Kp, TBM) || !make_map(&mm, Ab, Mp, Kp, tn)) return HELM_CUDA_ERROR;
    const cudaError_t e = tn == 128  ? gemm_tc<128, 2>(mn, mm, M, N, Kp, alpha, beta, C, ldc, s)
                          : tn == 64 ? gemm_tc<64, 3>(mn, mm, M, N, Kp, alpha, beta, C, ldc, s)
                          : tn == 32 ? gemm_tc<32, 3>(mn, mm, M, N, Kp, alpha, beta, C, ldc, s)
                                     : gemm_tc<16, 4>(mn, mm, M, N, Kp, alpha, beta, C, ldc, s);
    if (ordered) {
        if (cudaEventRecord(w.ev, s) != cudaSuccess) return HELM_CUDA_ERROR;
        w.used = true;
    }
    return e == cudaSuccess ? HELM_OK : HELM_CUDA_ERROR;
}

extern "C" helm_status nn_gemm_bf16_status(int* timed_out) {
    if (!timed_out) return HELM_BAD_ARG;
    int v = 0;
    if (cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(int)) != cudaSuccess) return HELM_CUDA_ERROR;
    *timed_out = v;
    if (v) {
        const int z = 0;
        if (cudaMemcpyToSymbol(g_tc_error, &z, sizeof(int)) != cudaSuccess) return HELM_CUDA_ERROR;
    }
    return HELM_OK;
}
