// Fused BLAS-1 and the scalar recurrences of BiCGStab and FGMRES.
//
// Reductions are deterministic: a fixed grid of kRedBlocks blocks writes one
// partial per block, and a single block sums the partials in a fixed order.
// Scalars (rho, alpha, omega, beta, norms, Hessenberg columns, Givens
// rotations) stay in device memory; the host only reads a status word.
#include <algorithm>

#include "bicg.cuh"
#include "helm_internal.cuh"

namespace helm {

namespace {

constexpr int TB = 256;

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double2 warp_sum(double2 v) {
    v.x = warp_sum(v.x);
    v.y = warp_sum(v.y);
    return v;
}

__global__ void __launch_bounds__(TB) k_dot(const double2* __restrict__ a, const double2* __restrict__ b,
                                            long long N, double2* partials) {
    pdl_begin();
    double2 acc = make_double2(0, 0);
    for (long long l = blockIdx.x * (long long)TB + threadIdx.x; l < N; l += (long long)gridDim.x * TB) {
        acc = cfmac(a[l], b[l], acc);
    }
    double v[2] = {acc.x, acc.y};
    block_tree<2>(v, threadIdx.x);
    if (threadIdx.x == 0) partials[blockIdx.x] = make_double2(v[0], v[1]);
}

__global__ void __launch_bounds__(TB) k_norm2(const double2* __restrict__ a, long long N, double* partials,
                                              double* out, unsigned* counter) {
    pdl_begin();
    double acc[1] = {0.0};
    for (long long l = blockIdx.x * (long long)TB + threadIdx.x; l < N; l += (long long)gridDim.x * TB)
        acc[0] = cnorm2(a[l], acc[0]);
    block_tree<1>(acc, threadIdx.x);
    if (threadIdx.x == 0) partials[blockIdx.x] = acc[0];
    if (norm_block_done(counter, gridDim.x)) {
        sum_parts<1>(partials, gridDim.x, threadIdx.x, acc);
        if (threadIdx.x == 0) *out = acc[0];
    }
}

// fixed-order sum of partials by one block of kFinThreads threads
template <typename T>
__device__ __forceinline__ T fin_sum(const T* partials, int nparts);

__device__ __forceinline__ double fin_sum_d(const double* p, int nparts) {
    __shared__ double red[kFinThreads / 32];
    double v = 0;
    for (int i = threadIdx.x; i < nparts; i += kFinThreads) v += p[i];
    v = warp_sum(v);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        v = red[lane];
        v = warp_sum(v);
    }
    __syncthreads();
    return v;  // valid in thread 0
}

__device__ __forceinline__ double2 fin_sum_c(const double2* p, int nparts, int stride = 1, int offset = 0) {
    __shared__ double2 red[kFinThreads / 32];
    double2 v = make_double2(0, 0);
    for (int i = threadIdx.x; i < nparts; i += kFinThreads) {
        double2 q = p[(long long)i * stride + offset];
        v.x += q.x;
        v.y += q.y;
    }
    v = warp_sum(v);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        v = red[lane];
        v = warp_sum(v);
    }
    __syncthreads();
    return v;
}

__global__ void __launch_bounds__(kFinThreads) k_sum_real(const double* partials, int nparts, double* out) {
    pdl_begin();
    double v = fin_sum_d(partials, nparts);
    if (threadIdx.x == 0) *out = v;
}
// ---------------------------------------------------------------- BiCGStab

__global__ void __launch_bounds__(TB) k_bicg_p(const double2* __restrict__ r, const double2* __restrict__ v,
                                               double2* __restrict__ p, const double2* __restrict__ sc, long long N) {
    pdl_begin();
    const double2 beta = sc[S_BETA], omega = sc[S_OMEGA];
    for (long long l = blockIdx.x * (long long)TB + threadIdx.x; l < N; l += (long long)gridDim.x * TB) {
        p[l] = cfma(beta, cfma(make_double2(-omega.x, -omega.y), v[l], p[l]), r[l]);
    }
}

// s = r - alpha v with ||s||^2, the scalar update in the last block
__global__ void __launch_bounds__(kFusedThreads) k_bicg_s_fused(const double2* __restrict__ r, const double2* __restrict__ v,
                                                                double2* __restrict__ s, double2* sc, long long N,
                                                                double* parts, unsigned* counter, double tol_abs) {
    pdl_begin();
    const double2 na = make_double2(-sc[S_ALPHA].x, -sc[S_ALPHA].y);
    double acc[1] = {0.0};
    for (long long l = blockIdx.x * (long long)kFusedThreads + threadIdx.x; l < N; l += (long long)gridDim.x * kFusedThreads) {
        const double2 q = cfma(na, v[l], r[l]);
        s[l] = q;
        acc[0] = cnorm2(q, acc[0]);
    }
    block_tree<1>(acc, threadIdx.x);
    if (threadIdx.x == 0) parts[blockIdx.x] = acc[0];
    if (last_block_done(counter, gridDim.x)) {
        double tot[1];
        sum_parts<1>(parts, gridDim.x, threadIdx.x, tot);
        if (threadIdx.x == 0) {
            bicg_snorm(sc, tot[0], tol_abs);
            *counter = 0;
        }
    }
}

// x += alpha phat + omega shat; r = s - omega t; ||r||^2 and the next rho = <rhat, r>
// with beta, in the last block (breakdown flag 3: rho = 0 for the next iteration)
__global__ void __launch_bounds__(kFusedThreads) k_bicg_xr_fused(double2* __restrict__ x, double2* __restrict__ r,
                                                                 const double2* __restrict__ phat,
                                                                 const double2* __restrict__ shat,
                                                                 const double2* __restrict__ s,
                                                                 const double2* __restrict__ t,
                                                                 const double2* __restrict__ rhat, double2* sc,
                                                                 long long N, double* parts, unsigned* counter,
                                                                 double tol, double bnorm) {
    pdl_begin();
    const double2 alpha = sc[S_ALPHA], omega = sc[S_OMEGA];
    const bool skip = sc[S_FLAGS].y == 1.0 || sc[S_STOP].x != 0.0;
    double rn = 0;
    double2 rho = make_double2(0, 0);
    for (long long l = blockIdx.x * (long long)kFusedThreads + threadIdx.x; l < N && !skip;
         l += (long long)gridDim.x * kFusedThreads) {
        x[l] = cfma(omega, shat[l], cfma(alpha, phat[l], x[l]));
        const double2 q = cfma(make_double2(-omega.x, -omega.y), t[l], s[l]);
        r[l] = q;
        rn = cnorm2(q, rn);
        rho = cfmac(rhat[l], q, rho);
    }
    double v[3] = {rn, rho.x, rho.y};
    block_tree<3>(v, threadIdx.x);
    if (threadIdx.x == 0) {
        parts[3 * blockIdx.x + 0] = v[0];
        parts[3 * blockIdx.x + 1] = v[1];
        parts[3 * blockIdx.x + 2] = v[2];
    }
    if (last_block_done(counter, gridDim.x)) {
        double tot[3];
        sum_parts<3>(parts, gridDim.x, threadIdx.x, tot);
        if (threadIdx.x == 0) {
            if (!skip) {
                bicg_rnorm(sc, tot[0]);
                bicg_rho_beta(sc, make_double2(tot[1], tot[2]), 3.0);
            }
            if (sc[S_STOP].x == 0.0) {
                const double res = sqrt(sc[S_RN2].x) / bnorm;
                if (sc[S_FLAGS].y != 0.0 || !isfinite(res) || res <= tol) sc[S_STOP].x = 1.0;
            }
            *counter = 0;
        }
    }
}

// recipes: 0 = rho & beta (complex partials), 1 = alpha, 2 = ||s||^2, 3 = omega, 4 = ||r||^2, 5 = reset
__global__ void __launch_bounds__(kFinThreads) k_bicg_scalar(int recipe, const double* partials, int nparts,
                                                             double2* sc, double tol_abs) {
    pdl_begin();
    if (recipe == 0 || recipe == 1) {
        double2 d = fin_sum_c(reinterpret_cast<const double2*>(partials), nparts);
        if (threadIdx.x != 0) return;
        if (recipe == 0) {
            sc[S_RHO] = d;
            if (d.x == 0 && d.y == 0) sc[S_FLAGS].y = 1;
            double2 q = cmul(cdiv(d, sc[S_RHO_OLD]), cdiv(sc[S_ALPHA], sc[S_OMEGA]));
            sc[S_BETA] = q;
            sc[S_FLAGS].x = 0;
        } else {
            if (d.x == 0 && d.y == 0) {
                sc[S_FLAGS].y = 1;
                sc[S_ALPHA] = make_double2(0, 0);
            } else {
                sc[S_ALPHA] = cdiv(sc[S_RHO], d);
            }
        }
    } else if (recipe == 2 || recipe == 4) {
        double v = fin_sum_d(partials, nparts);
        if (threadIdx.x != 0) return;
        if (recipe == 2) {
            sc[S_SN2] = make_double2(v, 0);
            if (sqrt(v) <= tol_abs) sc[S_FLAGS].x = 1;
        } else {
            sc[S_RN2] = make_double2(v, 0);
            if (sc[S_FLAGS].x == 0) sc[S_RHO_OLD] = sc[S_RHO];
        }
    } else if (recipe == 3) {
        double2 ts = fin_sum_c(reinterpret_cast<const double2*>(partials), nparts, 2, 0);
        double2 tt = fin_sum_c(reinterpret_cast<const double2*>(partials), nparts, 2, 1);
        if (threadIdx.x != 0) return;
        sc[S_TS] = ts;
        sc[S_TT] = tt;
        if (sc[S_FLAGS].x != 0) {
            sc[S_OMEGA] = make_double2(0, 0);
        } else if (tt.x == 0) {
            sc[S_FLAGS].y = 1;
            sc[S_OMEGA] = make_double2(0, 0);
        } else {
            double2 om = make_double2(ts.x / tt.x, ts.y / tt.x);
            sc[S_OMEGA] = om;
            if (om.x == 0 && om.y == 0) sc[S_FLAGS].y = 2;   // breakdown after this update
        }
    } else if (recipe == 5) {
        if (threadIdx.x != 0) return;
        sc[S_RHO_OLD] = make_double2(1, 0);
        sc[S_ALPHA] = make_double2(1, 0);
        sc[S_OMEGA] = make_double2(1, 0);
        sc[S_FLAGS] = make_double2(0, 0);
        sc[S_STOP] = make_double2(0, 0);
    }
}

// ------------------------------------------------------------------ FGMRES
// w += sign * sum_i V_i coef_i (the solution update of FGMRES)
__global__ void __launch_bounds__(TB) k_mupdate(const double2* __restrict__ V, int nv, const double2* __restrict__ coef,
                                                double sign, double2* __restrict__ w, long long N) {
    pdl_begin();
    __shared__ double2 c[kMaxRestart + 1];
    for (int i = threadIdx.x; i < nv; i += TB) c[i] = cscale(sign, coef[i]);
    __syncthreads();
    for (long long l = blockIdx.x * (long long)TB + threadIdx.x; l < N; l += (long long)gridDim.x * TB) {
        double2 s = w[l];
#pragma unroll 4
        for (int i = 0; i < nv; ++i) {
            s = cfma(c[i], V[(long long)i * N + l], s);
        }
        w[l] = s;
    }
}

// w += sign * sum_i V_i coef_i with complex64 vectors V (FP64 accumulation)
__global__ void __launch_bounds__(TB) k_mupdate32(const float2* __restrict__ V, int nv, const double2* __restrict__ coef,
                                                  double sign, double2* __restrict__ w, long long N) {
    pdl_begin();
    __shared__ double2 c[kMaxRestart + 1];
    for (int i = threadIdx.x; i < nv; i += TB) c[i] = cscale(sign, coef[i]);
    __syncthreads();
    for (long long l = blockIdx.x * (long long)TB + threadIdx.x; l < N; l += (long long)gridDim.x * TB) {
        double2 s = w[l];
#pragma unroll 4
        for (int i = 0; i < nv; ++i) {
            float2 vf = V[(long long)i * N + l];
            s = cfma(c[i], make_double2(vf.x, vf.y), s);
        }
        w[l] = s;
    }
}

__global__ void __launch_bounds__(TB) k_set_masked(double2* __restrict__ x, const double2* __restrict__ f,
                                                   const uint8_t* __restrict__ mask, long long N) {
    pdl_begin();
    for (long long l = blockIdx.x * (long long)TB + threadIdx.x; l < N; l += (long long)gridDim.x * TB)
        if (mask[l]) x[l] = f[l];
}

__global__ void __launch_bounds__(TB) k_cvt64to32(const double2* __restrict__ a, float2* __restrict__ b, long long N) {
    pdl_begin();
    for (long long l = blockIdx.x * (long long)TB + threadIdx.x; l < N; l += (long long)gridDim.x * TB)
        b[l] = make_float2((float)a[l].x, (float)a[l].y);
}
__global__ void __launch_bounds__(TB) k_cvt32to64(const float2* __restrict__ a, double2* __restrict__ b, long long N) {
    pdl_begin();
    for (long long l = blockIdx.x * (long long)TB + threadIdx.x; l < N; l += (long long)gridDim.x * TB)
        b[l] = make_double2((double)a[l].x, (double)a[l].y);
}

int stream_blocks(long long N) {
    long long b = (N + TB - 1) / TB;
    return (int)(b < 4 * kRedBlocks ? (b < 1 ? 1 : b) : 4 * kRedBlocks);
}

}  // namespace

void launch_dot(const double2* a, const double2* b, long long N, double2* partials, cudaStream_t s) {
    launch_after(k_dot, kRedBlocks, TB, 0, s, a, b, N, partials);
}
void launch_norm2(const double2* a, long long N, double* partials, double* out, unsigned* counters, cudaStream_t s) {
    // (no more blocks than the vector fills: each costs the last one a partial)
    const unsigned nb = (unsigned)std::min<long long>(kRedBlocks, (N + TB - 1) / TB);
    launch_after(k_norm2, nb, TB, 0, s, a, N, partials, out, counters + kNormVector);
}
void launch_sum_real(const double* partials, int nparts, double* out, cudaStream_t s) {
    launch_after(k_sum_real, 1, kFinThreads, 0, s, partials, nparts, out);
}
void launch_bicg_update_p(const double2* r, const double2* v, double2* p, const double2* sc, long long N,
                          cudaStream_t s) {
    launch_after(k_bicg_p, stream_blocks(N), TB, 0, s, r, v, p, sc, N);
}
void launch_bicg_s_fused(const double2* r, const double2* v, double2* sv, double2* sc, long long N, double* parts,
                         unsigned* counter, double tol_abs, cudaStream_t s) {
    launch_after(k_bicg_s_fused, kRedBlocks, kFusedThreads, 0, s, r, v, sv, sc, N, parts, counter, tol_abs);
}
void launch_bicg_xr_fused(double2* x, double2* r, const double2* phat, const double2* shat, const double2* sv,
                          const double2* t, const double2* rhat, double2* sc, long long N, double* parts,
                          unsigned* counter, double tol, double bnorm, cudaStream_t s) {
    launch_after(k_bicg_xr_fused, kRedBlocks, kFusedThreads, 0, s, x, r, phat, shat, sv, t, rhat, sc, N, parts, counter, tol,
                                                         bnorm);
}
void launch_bicg_scalar(int recipe, const double* partials, int nparts, double2* sc, double tol_abs,
                        cudaStream_t s) {
    launch_after(k_bicg_scalar, 1, kFinThreads, 0, s, recipe, partials, nparts, sc, tol_abs);
}
void launch_mupdate(const double2* V, int nv, const double2* coef, double sign, double2* w, long long N,
                    cudaStream_t s) {
    launch_after(k_mupdate, stream_blocks(N), TB, 0, s, V, nv, coef, sign, w, N);
}
void launch_mupdate32(const float2* V, int nv, const double2* coef, double sign, double2* w, long long N,
                      cudaStream_t s) {
    launch_after(k_mupdate32, stream_blocks(N), TB, 0, s, V, nv, coef, sign, w, N);
}
void launch_set_masked(double2* x, const double2* f, const uint8_t* mask, long long N, cudaStream_t s) {
    launch_after(k_set_masked, stream_blocks(N), TB, 0, s, x, f, mask, N);
}
void launch_cvt_f64_to_f32(const double2* a, float2* b, long long N, cudaStream_t s) {
    launch_after(k_cvt64to32, stream_blocks(N), TB, 0, s, a, b, N);
}
void launch_cvt_f32_to_f64(const float2* a, double2* b, long long N, cudaStream_t s) {
    launch_after(k_cvt32to64, stream_blocks(N), TB, 0, s, a, b, N);
}

}  // namespace helm
