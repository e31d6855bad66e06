// The Arnoldi step of FGMRES: classical Gram-Schmidt applied twice, the Givens rotation
// of the new Hessenberg column and the normalised basis vector, in four launches:
//
//   k_gs<DOT>     h = V^H w                                     (H column = h)
//   k_gs<UPDOT>   w -= V h;  h2 = V^H w                         (H column += h2)
//   k_gs<UPNORM>  w -= V h2; ||w||^2; Givens rotation, estimate of the residual
//   k_gs_scale    v = w / ||w||, and its complex64 copy for a complex64 preconditioner
//
// What bounds them: the FP64 pipe (2 instructions per clock and SM; four multiply-adds per
// basis entry and pass) on grids of 10^5 nodes and more, the launches and the serial
// tail on the small ones.  So a reduction must not spend FP64 instructions on idle
// lanes: a tile of V is staged in shared memory (asynchronous copies), the update reads
// it with one lane per row and the dots read it with one lane per basis vector, each
// thread adding its own rows in a register, and only at the end of a block do the
// threads of one vector meet in a shared-memory tree.  (A butterfly of warp shuffles per
// vector costs 10 FP64 instructions of 32 lanes for 31 useful additions; with one row
// per lane, as on 64 x 64 nodes, that was 2.5 times the dot's own arithmetic.)  Staging
// also lets w -= V h and V^H w read V once.  Rows per tile: 32 on small grids, so that
// 4096 nodes use 128 SMs instead of 8, up to 256 where shared memory allows.
//
// Measured (ncu, cold, one step; before: nine launches): 64^2 nodes, 8 vectors on average,
// 75 -> 38 us; 48^3 to 96^3 nodes, 3.5 vectors, 115 -> 81 us.  Sums are in a fixed order:
// deterministic.
#include <algorithm>

#include "bicg.cuh"
#include "helm_internal.cuh"

namespace helm {

namespace {

constexpr int GT = 256;              // threads
enum { GS_DOT = 0, GS_UPDOT = 1, GS_UPNORM = 2 };

struct GivensArgs {
    double2* H;                      // column-major Hessenberg matrix, ldh rows
    int ldh, j;
    double* cs;
    double2* sn;
    double2* g;
    double* wnorm2;                  // ||w||^2, and in the next entry 1 / ||w|| (0 for w = 0)
    double* est;                     // |g_{j+1}|: the residual's norm
};

__device__ __forceinline__ void gs_copy16(void* dst, const void* src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// red[q nv + v] (q < ng) summed over q into red[v], pairwise; every thread of the block
// calls it, thread t holding entry t (t < ng nv)
__device__ __forceinline__ void tree(double2* red, int t, int nv, int ng) {
    const int q = t / nv;
    for (int n = ng; n > 1;) {
        const int half = (n + 1) >> 1;
        __syncthreads();
        if (q < n - half) red[t] = cadd(red[t], red[t + half * nv]);
        n = half;
    }
    __syncthreads();
}

// (2^-e, 2^e), e the binary exponent of z's larger part (kept where both are normal numbers;
// 0 for a part that is not finite)
__device__ __forceinline__ double2 pow2_scale(double2 z) {
    int e = max(__double2hiint(z.x) & 0x7fffffff, __double2hiint(z.y) & 0x7fffffff) >> 20;
    e = e == 2047 ? 1023 : min(max(e, 1), 2045);
    return make_double2(__hiloint2double((2046 - e) << 20, 0), __hiloint2double(e << 20, 0));
}

// Givens step for column j; the column and the earlier rotations are staged in shared
// memory first (thread 0 walks them in a dependent chain: with each entry loaded from
// memory inside the chain a step took 12 us at j = 7 and grew with j)
__device__ void givens(const GivensArgs& a, double wn2, double2* col, double2* sn, double* cs) {
    const int t = threadIdx.x, j = a.j;
    double2* Hc = a.H + (long long)j * a.ldh;
    for (int i = t; i <= j; i += GT) {
        col[i] = Hc[i];
        if (i < j) {
            sn[i] = a.sn[i];
            cs[i] = a.cs[i];
        }
    }
    __syncthreads();
    if (t == 0) {
        double2 x = col[0];
        for (int i = 0; i < j; ++i) {
            const double2 b = col[i + 1], s = sn[i];
            const double c = cs[i];
            col[i] = cfma(s, b, cscale(c, x));
            x = cfmac(make_double2(-s.x, -s.y), x, cscale(c, b));
        }
        // c = |x| / t, s = (x / |x|) ||w|| / t, r = (x / |x|) t with t^2 = |x|^2 + ||w||^2; the
        // square roots do not wait for one another (a hypot or a division apiece cost this
        // one thread about a microsecond each).  |x| and x / |x| come from x scaled to about
        // 1, as hypot does it: below 1e-154 |x|^2 would lose its digits
        const double2 sx = pow2_scale(x), xs = cscale(sx.x, x);
        const double as2 = xs.x * xs.x + xs.y * xs.y, t2 = x.x * x.x + x.y * x.y + wn2;
        const double ias = rsqrt(as2), it = rsqrt(t2), hn = wn2 * rsqrt(wn2);
        double c;
        double2 s, r;
        if (wn2 == 0) {
            c = 1; s = make_double2(0, 0); r = x;
        } else if (as2 == 0) {
            c = 0; s = make_double2(1.0, 0.0); r = make_double2(hn, 0);
        } else {
            const double2 ph = cscale(ias, xs);
            c = as2 * ias * sx.y * it;
            s = cscale(hn * it, ph);
            r = cscale(t2 * it, ph);
        }
        a.cs[j] = c;
        a.sn[j] = s;
        col[j] = r;
        const double2 gj = a.g[j], gn = cscale(-1.0, cmulc(s, gj));
        a.g[j + 1] = gn;
        a.g[j] = cscale(c, gj);
        const double2 sg = pow2_scale(gn), gs = cscale(sg.x, gn);
        *a.est = sqrt(gs.x * gs.x + gs.y * gs.y) * sg.y;
        a.wnorm2[0] = wn2;
        a.wnorm2[1] = wn2 == 0 ? 0.0 : rsqrt(wn2);
    }
    __syncthreads();
    for (int i = t; i <= j; i += GT) Hc[i] = col[i];
    if (t == 0) Hc[j + 1] = make_double2(0, 0);
}

// W32 (DOT only): w is given in complex64 (w32) and written in complex128 on the way
template <int MODE, bool W32>
__global__ void __launch_bounds__(GT) k_gs(const double2* __restrict__ V, int nv, long long N,
                                           const float2* __restrict__ w32, double2* w, const double2* __restrict__ coef,
                                           int lrt, double2* partials, unsigned* counter, double2* Hcol,
                                           double2* coef_out, GivensArgs ga) {
    pdl_begin();
    extern __shared__ double2 gs_smem[];
    const int RT = 1 << lrt, t = threadIdx.x;
    double2* vs = gs_smem;                                 // [nv][RT + 1]
    double2* ws = vs + nv * (RT + 1);                      // [RT]
    double2* red = ws + RT;                                // [GT]
    double2* cf = red + GT;                                // [nv]
    const int own = t & (RT - 1), ig = t >> lrt, IG = GT >> lrt;
    const int ng = GT / nv, vi = t % nv, rg = t / nv;      // dots: vector vi, rows rg, rg + ng, ...
    if (MODE != GS_DOT)
        for (int i = t; i < nv; i += GT) cf[i] = cscale(-1.0, coef[i]);
    double2 acc = make_double2(0, 0);
    for (long long t0 = (long long)blockIdx.x * RT; t0 < N; t0 += (long long)gridDim.x * RT) {
        const int rows = (int)min((long long)RT, N - t0);
        __syncthreads();                                   // the previous tile is consumed
        for (int e = t; e < nv << lrt; e += GT) {
            const int i = e >> lrt, r = e & (RT - 1);
            gs_copy16(vs + i * (RT + 1) + r, r < rows ? V + HCHK((long long)i * N + t0 + r, (long long)nv * N) : V, r < rows);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        double2 wv = make_double2(0, 0);
        if (ig == 0 && own < rows) {
            if (W32) {
                const float2 q = w32[HCHK(t0 + own, N)];
                wv = make_double2(q.x, q.y);
                w[HCHK(t0 + own, N)] = wv;
            } else {
                wv = w[HCHK(t0 + own, N)];
            }
        }
        if (MODE == GS_DOT && ig == 0) ws[own] = wv;
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
        if (MODE != GS_DOT) {
            double2 s = ig == 0 ? wv : make_double2(0, 0);
#pragma unroll 4
            for (int i = ig; i < nv; i += IG) s = cfma(cf[i], vs[i * (RT + 1) + own], s);
            if (IG > 1) {
                red[t] = s;
                __syncthreads();
                if (ig == 0)
                    for (int q = 1; q < IG; ++q) s = cadd(s, red[q * RT + own]);
            }
            if (ig == 0) {
                if (own < rows) w[HCHK(t0 + own, N)] = s;
                if (MODE == GS_UPDOT) ws[own] = s;
                else acc.x = cnorm2(s, acc.x);             // (zero past the last row)
            }
            if (MODE == GS_UPDOT) __syncthreads();
        }
        if (MODE != GS_UPNORM && rg < ng) {
#pragma unroll 4
            for (int r = rg; r < rows; r += ng) acc = cfmac(vs[vi * (RT + 1) + r], ws[r], acc);
        }
    }
    const int nr = MODE == GS_UPNORM ? 1 : nv, nq = MODE == GS_UPNORM ? GT : ng;
    __syncthreads();
    red[t] = acc;
    tree(red, t, nr, nq);
    if (t < nr) partials[(long long)blockIdx.x * nr + t] = red[t];
    if (!last_block_done(counter, gridDim.x)) return;
    // the last block: the blocks' sums, then the scalars that follow from them
    acc = make_double2(0, 0);
    if (t < nr * nq)
#pragma unroll 8
        for (unsigned b = t / nr; b < gridDim.x; b += nq) acc = cadd(acc, __ldcg(partials + (long long)b * nr + t % nr));
    red[t] = acc;
    tree(red, t, nr, nq);
    if (MODE != GS_UPNORM) {
        if (t < nv) {
            const double2 h = red[t];
            Hcol[t] = MODE == GS_DOT ? h : cadd(Hcol[t], h);
            coef_out[t] = h;
        }
    } else {
        // (the staged tile is done with: its space holds the column and the rotations)
        const double wn2 = red[0].x;
        double2* col = vs;
        givens(ga, wn2, col, col + ga.j + 1, reinterpret_cast<double*>(col + 2 * ga.j + 2));
    }
    if (t == 0) *counter = 0;
}

// v = w / ||w|| (unchanged when it is 0), and v32 = complex64(v) if given.  norm: ||w||^2,
// and with g == null also 1 / ||w||; with g, g = (||w||, 0, ...) of m1 entries (the start of
// a restart cycle)
__global__ void __launch_bounds__(256) k_gs_scale(const double2* w, double2* v, float2* __restrict__ v32,
                                                  const double* __restrict__ norm, long long N, double2* g, int m1) {
    pdl_begin();
    double inv;
    if (g) {
        const double nn = sqrt(norm[0]);
        if (blockIdx.x == 0 && (int)threadIdx.x < m1) g[threadIdx.x] = make_double2(threadIdx.x == 0 ? nn : 0.0, 0);
        inv = nn == 0 ? 0.0 : 1.0 / nn;
    } else {
        inv = norm[1];
    }
    if (inv == 0) return;
    for (long long l = blockIdx.x * 256LL + threadIdx.x; l < N; l += gridDim.x * 256LL) {
        const double2 q = cscale(inv, w[HCHK(l, N)]);
        v[HCHK(l, N)] = q;
        if (v32) v32[HCHK(l, N)] = make_float2((float)q.x, (float)q.y);
    }
}

// y = R^-1 g for the k x k upper triangle R of H, in shared memory, column by column: each
// y_i is subtracted from the remaining right-hand side by all threads (one thread
// walking memory took 54 us at k = 15)
__global__ void __launch_bounds__(64) k_hsolve(const double2* __restrict__ H, int ldh, int k, const double2* __restrict__ g,
                                               double2* __restrict__ y) {
    pdl_begin();
    extern __shared__ double2 hs_smem[];
    double2* R = hs_smem;                                  // [k][k] column-major
    double2* b = hs_smem + k * k;
    for (int e = threadIdx.x; e < k * k; e += 64) R[e] = H[(long long)(e / k) * ldh + e % k];
    for (int i = threadIdx.x; i < k; i += 64) b[i] = g[i];
    __syncthreads();
    for (int i = k - 1; i >= 0; --i) {
        if (threadIdx.x == 0) {
            b[i] = cdiv(b[i], R[i * k + i]);
            y[i] = b[i];
        }
        __syncthreads();
        const double2 yi = b[i];
        for (int q = threadIdx.x; q < i; q += 64) b[q] = cfma(make_double2(-yi.x, -yi.y), R[i * k + q], b[q]);
        __syncthreads();
    }
}

// rows per tile (log2): as many as 66 KB of staged vectors allow, fewer while the grid
// would have under two tiles per SM
int gs_lrt(int nv, long long N) {
    int l = nv <= 15 ? 8 : nv <= 31 ? 7 : 6;
    while (l > 5 && ((N + (1 << l) - 1) >> l) < 2 * 152) --l;
    return l;
}

size_t gs_smem_bytes(int nv, int lrt) { return ((size_t)nv * ((1 << lrt) + 2) + (1 << lrt) + GT) * sizeof(double2); }

template <int MODE, bool W32>
cudaError_t gs(const double2* V, int nv, long long N, const float2* w32, double2* w, const double2* coef, double2* partials,
               unsigned* counter, double2* Hcol, double2* coef_out, const GivensArgs& ga, cudaStream_t s) {
    const int lrt = gs_lrt(nv, N);
    const size_t smem = gs_smem_bytes(nv, lrt);            // (the tail's 5 doubles a row of H fit into the tile)
    if (smem > 48 * 1024) {
        const cudaError_t e =
            cudaFuncSetAttribute(k_gs<MODE, W32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
        if (e != cudaSuccess) return e;
    }
    const long long tiles = (N + (1 << lrt) - 1) >> lrt;
    // a tile is loaded, then used: another block on the SM fills the wait (two; with more the
    // last block's sums over the blocks cost what the overlap gains)
    const unsigned nb = (unsigned)std::min<long long>(tiles, kRedBlocks);
    launch_after(k_gs<MODE, W32>, nb, GT, smem, s, V, nv, N, w32, w, coef, lrt, partials, counter, Hcol, coef_out, ga);
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_arnoldi(const double2* V, int j, long long N, const float2* w32, double2* w, double2* H, int ldh,
                           double* cs, double2* sn, double2* g, double2* coef, double* wnorm2, double* est,
                           double2* partials, unsigned* counter, float2* v32, cudaStream_t s) {
    const int nv = j + 1;
    double2 *Hcol = H + (long long)j * ldh, *c1 = coef, *c2 = coef + kMaxRestart + 1;
    const GivensArgs ga{H, ldh, j, cs, sn, g, wnorm2, est};
    cudaError_t e = w32 ? gs<GS_DOT, true>(V, nv, N, w32, w, nullptr, partials, counter, Hcol, c1, ga, s)
                        : gs<GS_DOT, false>(V, nv, N, nullptr, w, nullptr, partials, counter, Hcol, c1, ga, s);
    if (e == cudaSuccess) e = gs<GS_UPDOT, false>(V, nv, N, nullptr, w, c1, partials, counter, Hcol, c2, ga, s);
    if (e == cudaSuccess) e = gs<GS_UPNORM, false>(V, nv, N, nullptr, w, c2, partials, counter, Hcol, nullptr, ga, s);
    if (e == cudaSuccess) launch_gs_scale(w, w, v32, wnorm2, N, nullptr, 0, s);
    return e;
}

void launch_gs_scale(const double2* w, double2* v, float2* v32, const double* norm2, long long N, double2* g, int m1,
                     cudaStream_t s) {
    const long long b = (N + 255) / 256;
    launch_after(k_gs_scale, (unsigned)std::min<long long>(b, 4 * kRedBlocks), 256, 0, s, w, v, v32, norm2, N, g, m1);
}

cudaError_t launch_hsolve(const double2* H, int ldh, int k, const double2* g, double2* y, cudaStream_t s) {
    const size_t smem = ((size_t)k * k + k) * sizeof(double2);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k_hsolve, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (kMaxRestart * kMaxRestart + kMaxRestart) * (int)sizeof(double2));
        if (e != cudaSuccess) return e;
    }
    launch_after(k_hsolve, 1, 64, smem, s, H, ldh, k, g, y);
    return cudaSuccess;
}

}  // namespace helm
