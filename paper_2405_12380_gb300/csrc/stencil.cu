// Matrix-free Helmholtz operator, residual and relaxation sweeps (Eq. 1-2).
//
// Blocks of 256 threads: 32 x 8 over (x, y), or (complex128, odd and 2D grids) 256 nodes or
// node pairs in the flat order.  Per node two byte tables (neighbour code,
// layer index) replace the mask loads and the index arithmetic; k^2 and 1/diag
// come from per-layer tables in Op (or the stored field).  Kernel families:
//   k_apply_z        3D operator/residual marching in z (planes in registers,
//                    x-neighbours by warp shuffles), complex128 and complex64
//   k_march_c64      3D complex64 operator and damped Jacobi, two nodes per thread; the
//                    red rows' residual; the operator with the partial sums of a
//                    BiCGStab scalar (DOT)
//   k_rbgs_c64       3D complex64 red-black half-sweep, two nodes per thread
//   k_sweep_c64      3D complex64 full red-black sweep in one launch (old planes
//                    staged in shared memory by cp.async, halo rows recomputed)
//   k_apply, k_jacobi, k_rbgs   the general forms (2D, no tables, complex128)
//   k_jacobi_tile    several 2D Jacobi sweeps per launch (small grids)
//   k_apply_bicg(_df)           the BiCGStab operator with its fused reduction
//   k_cycle_df       the red-black part of the FP64 trunk-basis hybrid cycle in
//                    double-float arithmetic, one cooperative launch
// FP64 is the scarce pipe on GB300 (2 instructions per clock per SM against 128
// for FP32), so the FP64 path moves its sweeps onto FP32 pairs.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "bicg.cuh"
#include "helm_internal.cuh"

namespace helm {

namespace {

constexpr int BX = 32, BY = 8;
constexpr int kJacobiTileSweeps = 5;      // sweeps of one tiled Jacobi launch (at most 26^2 threads)

__device__ __forceinline__ int layer_index(int i, int n, int L) {
    int d = min(i, n - 1 - i);
    return max(0, L - d);
}

template <typename R>
__device__ __forceinline__ int node_layer(const Op<R>& op, int i, int j, int k) {
    int m = max(layer_index(i, op.n, op.L), layer_index(j, op.n, op.L));
    if (op.dim == 3) m = max(m, layer_index(k, op.n, op.L));
    return m;
}

template <typename R>
__device__ __forceinline__ typename CT<R>::T diag_of(const Op<R>& op, long long l, int m, int conj) {
    typename CT<R>::T d;
    if (op.k2) {
        d = op.k2[l];
        d.x -= op.dsub;
    } else {
        d.x = op.dre;
        d.y = op.im[m];
    }
    if (conj) d.y = -d.y;
    return d;
}

template <typename R>
__device__ __forceinline__ typename CT<R>::T invd_of(const Op<R>& op, long long l, int m, int conj) {
    typename CT<R>::T d = op.k2 ? op.invd[l] : op.invd_tab[m];
    if (conj) d.y = -d.y;
    return d;
}

// sum of the fluid neighbours of a fluid node; `code` is the node's neighbour code
// (bit q set: neighbour q is fluid, q = -x, +x, -y, +y, -z, +z), one byte load
// instead of six mask loads
template <typename R>
__device__ __forceinline__ typename CT<R>::T nbr_sum(const Op<R>& op, const typename CT<R>::T* __restrict__ x,
                                                     long long l, unsigned code) {
    using C = typename CT<R>::T;
    const long long sy = op.n, sz = (long long)op.n * op.n;
    C z;
    z.x = 0; z.y = 0;
    // pairwise (tree) sum: three independent adds, then two -- shorter FP64 dependency chains
    const C a = (code & 1u) ? x[HCHK(l - 1, op.N)] : z;
    const C b = (code & 2u) ? x[HCHK(l + 1, op.N)] : z;
    const C c = (code & 4u) ? x[HCHK(l - sy, op.N)] : z;
    const C d = (code & 8u) ? x[HCHK(l + sy, op.N)] : z;
    if (op.face) {
        // Sommerfeld / Neumann boundary rows: axis a weighs 2^-(b - [on an axis-a face])
        const unsigned fc = op.face[l];
        const int nb = (int)(fc >> 4);
        const R wx = ldexp((R)1, -(nb - (int)(fc & 1u))), wy = ldexp((R)1, -(nb - (int)((fc >> 1) & 1u)));
        C s = cadd(cscale(wx, cadd(a, b)), cscale(wy, cadd(c, d)));
        if (op.dim == 3) {
            const R wz = ldexp((R)1, -(nb - (int)((fc >> 2) & 1u)));
            const C e = (code & 16u) ? x[HCHK(l - sz, op.N)] : z;
            const C f = (code & 32u) ? x[HCHK(l + sz, op.N)] : z;
            s = cadd(s, cscale(wz, cadd(e, f)));
        }
        return s;
    }
    C s = cadd(cadd(a, b), cadd(c, d));
    if (op.dim == 3) {
        const C e = (code & 16u) ? x[HCHK(l - sz, op.N)] : z;
        const C f = (code & 32u) ? x[HCHK(l + sz, op.N)] : z;
        s = cadd(s, cadd(e, f));
    }
    return s;
}

constexpr unsigned kMasked = 0x80u;

// The end of a kernel that left one partial of ||r||^2 per block: the last block sums them
// in a fixed order into *out (no launch of its own; without a counter they are left).
struct NormTail {
    double* out;
    unsigned* counter;
};
__device__ __forceinline__ void norm_tail(const NormTail& t, const double* partials, unsigned nblocks, int tid) {
    if (!t.counter) return;
    if (norm_block_done(t.counter, nblocks)) {
        double v[1];
        sum_parts<1>(partials, (int)nblocks, tid, v);
        if (tid == 0) *t.out = v[0];
    }
}

// neighbour code and layer index of a node: from the handle's tables, or from the
// mask and the indices when the operator carries no tables (no-allocation path)
template <typename R>
__device__ __forceinline__ unsigned node_code(const Op<R>& op, long long l) {
    if (op.nbm) return op.nbm[l];
    if (op.mask[l]) return kMasked;
    const long long sy = op.n, sz = (long long)op.n * op.n;
    unsigned c = 0;
    if (!op.mask[l - 1]) c |= 1u;
    if (!op.mask[l + 1]) c |= 2u;
    if (!op.mask[l - sy]) c |= 4u;
    if (!op.mask[l + sy]) c |= 8u;
    if (op.dim == 3) {
        if (!op.mask[l - sz]) c |= 16u;
        if (!op.mask[l + sz]) c |= 32u;
    }
    return c;
}

template <typename R>
__device__ __forceinline__ int node_lidx(const Op<R>& op, long long l, int i, int j, int k) {
    return op.lidx ? (int)op.lidx[l] : node_layer(op, i, j, k);
}

template <typename R>
__device__ __forceinline__ void block_reduce_store(double v, double* out) {
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    int tid = threadIdx.x + blockDim.x * threadIdx.y;
    int lane = tid & 31, w = tid >> 5;
    if (lane == 0) red[w] = v;
    __syncthreads();
    int nw = (blockDim.x * blockDim.y) >> 5;
    if (w == 0) {
        v = lane < nw ? red[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) *out = v;
    }
}

// y = A x, or y = f - A x (resid), at one node; returns y_l
template <typename R, bool RESID>
__device__ __forceinline__ typename CT<R>::T apply_point(const Op<R>& op, const typename CT<R>::T* __restrict__ x,
                                              const typename CT<R>::T* __restrict__ f, typename CT<R>::T* __restrict__ y,
                                              int conj, int i, int j, int k, long long l) {
    using C = typename CT<R>::T;
    const C xc = x[l];
    const unsigned code = node_code(op, l);
    C out;
    if (code & kMasked) {
        out = xc;
    } else {
        const C s = nbr_sum(op, x, l, code);
        const C d = diag_of(op, l, node_lidx(op, l, i, j, k), conj);
        out.x = op.hinv2 * s.x + (d.x * xc.x - d.y * xc.y);
        out.y = op.hinv2 * s.y + (d.x * xc.y + d.y * xc.x);
    }
    if (RESID) out = csub(f[l], out);
    y[l] = out;
    return out;
}
__device__ __forceinline__ double norm_acc(double2 a, double s) { return cnorm2(a, s); }
__device__ __forceinline__ double norm_acc(float2 a, double s) { return s + ((double)a.x * a.x + (double)a.y * a.y); }

// 3D operator marching in z: a block owns 256 consecutive nodes of a plane (whatever rows
// they lie in, so that every lane has a node: with one row per warp a 129-node row filled
// four fifths of its lanes, and an FP64 instruction costs the same however few are active)
// and walks zc planes.  The z-neighbours come from registers (each plane of x is loaded
// once, two planes ahead of its use), the x-neighbours from warp shuffles (fluid nodes are
// interior, so theirs are the neighbours in the plane's order; the two ends of the warp
// load from memory), the y-neighbours from L1 or L2.  Bound by the FP64 pipe in complex128
// (16 instructions a node, 20 with the residual and its norm): the residual with its norm
// at 129^3 151 -> 99 us, 68 us at the pipe's rate.  (In 32 x 8 tiles, whose y-neighbours
// share an L1, the times are the same to 1% from 64^3 to 256^3.)
constexpr int AZ = 256;

template <typename R, bool RESID, bool NORM>
__global__ void __launch_bounds__(AZ) k_apply_z(Op<R> op, int zc, const typename CT<R>::T* __restrict__ x,
                                                const typename CT<R>::T* __restrict__ f,
                                                typename CT<R>::T* __restrict__ y, double* partials, int conj,
                                                NormTail tail) {
    pdl_begin();
    using C = typename CT<R>::T;
    const int sy = op.n, sz = op.n * op.n;                 // (N < 2^31)
    const int q = blockIdx.x * AZ + threadIdx.x;           // index in the plane
    const int k0 = blockIdx.y * zc;
    const int k1 = min(op.n, k0 + zc);
    const bool valid = q < sz;
    const int lane = threadIdx.x & 31;
    C zero;
    zero.x = 0; zero.y = 0;
    long long l = q + (long long)sz * k0;
    C prev = (valid && k0 > 0) ? x[HCHK(l - sz, op.N)] : zero;
    C cur = valid ? x[HCHK(l, op.N)] : zero;
    C next = (valid && k0 + 1 < op.n) ? x[HCHK(l + sz, op.N)] : zero;
    // the per-node tables are read one plane ahead as well, so that no load of
    // the loop is used in the iteration that issues it
    unsigned code = valid ? (unsigned)op.nbm[l] : kMasked;
    int li = valid ? (int)op.lidx[l] : 0;
    double acc = 0.0;
    for (int k = k0; k < k1; ++k, l += sz) {
        const bool more = valid && k + 1 < k1;
        const C next2 = (more && k + 2 < op.n) ? x[HCHK(l + 2 * sz, op.N)] : zero;
        const unsigned code_n = more ? (unsigned)op.nbm[HCHK(l + sz, op.N)] : kMasked;
        const int li_n = more ? (int)op.lidx[HCHK(l + sz, op.N)] : 0;
        C xm, xp, fv = zero;
        if (RESID && valid) fv = f[HCHK(l, op.N)];
        xm.x = __shfl_up_sync(0xffffffffu, cur.x, 1);
        xm.y = __shfl_up_sync(0xffffffffu, cur.y, 1);
        xp.x = __shfl_down_sync(0xffffffffu, cur.x, 1);
        xp.y = __shfl_down_sync(0xffffffffu, cur.y, 1);
        if (lane == 0 && (code & 1u)) xm = x[HCHK(l - 1, op.N)];
        if (lane == 31 && (code & 2u)) xp = x[HCHK(l + 1, op.N)];
        C out;
        if (code & kMasked) {
            out = cur;
        } else {
            const C a = (code & 1u) ? xm : zero;
            const C b = (code & 2u) ? xp : zero;
            const C c = (code & 4u) ? x[l - sy] : zero;
            const C d = (code & 8u) ? x[l + sy] : zero;
            const C e = (code & 16u) ? prev : zero;
            const C g = (code & 32u) ? next : zero;
            const C s = cadd(cadd(cadd(a, b), cadd(c, d)), cadd(e, g));
            const C dg = diag_of(op, l, li, conj);
            out.x = op.hinv2 * s.x + (dg.x * cur.x - dg.y * cur.y);
            out.y = op.hinv2 * s.y + (dg.x * cur.y + dg.y * cur.x);
        }
        if (valid) {
            if (RESID) out = csub(fv, out);
            y[HCHK(l, op.N)] = out;
            if (NORM) acc = norm_acc(out, acc);
        }
        prev = cur;
        cur = next;
        next = next2;
        code = code_n;
        li = li_n;
    }
    if (NORM) {
        double v[1] = {acc};
        block_tree<1>(v, threadIdx.x);
        if (threadIdx.x == 0) partials[blockIdx.x + gridDim.x * blockIdx.y] = v[0];
        norm_tail(tail, partials, gridDim.x * gridDim.y, threadIdx.x);
    }
}

// ---- complex64 in 3D: two consecutive x-nodes per thread, so that every vector
// access is one 16-byte load or store and a warp covers 64 nodes of a row.  Needs
// n even (every row starts on a 16-byte boundary) and 16-byte aligned vectors; the
// per-node tables are read as byte pairs.  Marches in z like k_apply_z, with the
// right-hand side prefetched one plane ahead too.  A pair whose two nodes have
// all six neighbours fluid (the common case) takes no selects.
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float2 pick(unsigned c, unsigned bit, float2 v) {
    return (c & bit) ? v : make_float2(0.f, 0.f);
}

// neighbour sums of the two nodes of a pair (same summation tree as k_apply_z)
__device__ __forceinline__ void pair_sums(unsigned c0, unsigned c1, float2 left, float2 right, float4 cur,
                                          float4 ym, float4 yp, float4 zm, float4 zp, float2& s0, float2& s1) {
    if ((c0 & c1) == 0x3Fu) {
        s0 = cadd(cadd(cadd(left, hi2(cur)), cadd(lo2(ym), lo2(yp))), cadd(lo2(zm), lo2(zp)));
        s1 = cadd(cadd(cadd(lo2(cur), right), cadd(hi2(ym), hi2(yp))), cadd(hi2(zm), hi2(zp)));
    } else {
        s0 = cadd(cadd(cadd(pick(c0, 1u, left), pick(c0, 2u, hi2(cur))),
                       cadd(pick(c0, 4u, lo2(ym)), pick(c0, 8u, lo2(yp)))),
                  cadd(pick(c0, 16u, lo2(zm)), pick(c0, 32u, lo2(zp))));
        s1 = cadd(cadd(cadd(pick(c1, 1u, lo2(cur)), pick(c1, 2u, right)),
                       cadd(pick(c1, 4u, hi2(ym)), pick(c1, 8u, hi2(yp)))),
                  cadd(pick(c1, 16u, hi2(zm)), pick(c1, 32u, hi2(zp))));
    }
}

// KIND 0: y = A x (FLAG: y = f - A x); KIND 1: damped-Jacobi sweep y = x + omega
// D^-1 (f - A x) (FLAG: from x = 0, x not read); KIND 2: the residual f - A x of the
// red node of each pair (colour 0), written compactly as one float2 per pair
// (zero on masked nodes)
// DOT (KIND 0 only): the BiCGStab reduction of launch_apply32_bicg in the epilogue,
// 1: conj(w) y (for alpha), 2: conj(y) w and |y|^2 (for omega); FP32 sums per
// thread and across the block in a fixed order, one partial per block
struct Dot32 {
    const float4* w;
    double2* sc;
    float* parts;
};

template <int KIND, bool FLAG, bool NORM, int DOT = 0>
__global__ void __launch_bounds__(BX * BY) k_march_c64(Op<float> op, int zc, float omega,
                                                       const float4* __restrict__ x, const float4* __restrict__ f,
                                                       float4* __restrict__ y, double* partials, int conj,
                                                       Dot32 dot = Dot32{}, NormTail tail = NormTail{}) {
    pdl_begin();
    static_assert(DOT == 0 || (KIND == 0 && !FLAG && !NORM), "the fused reduction follows y = A x only");
    constexpr bool NBR = !(KIND == 1 && FLAG);             // neighbours (and x) are read
    constexpr bool RHS = KIND >= 1 || FLAG;                // f is read
    constexpr unsigned kMM = kMasked | (kMasked << 8);
    const int n = op.n, h = n >> 1;
    const int i2 = blockIdx.x * BX + threadIdx.x;          // pair index within the row
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k0 = blockIdx.z * zc;
    const int k1 = min(n, k0 + zc);
    const bool valid = i2 < h && j < n;
    const int sy = h, sz = h * n;                          // strides in pairs (N < 2^31)
    [[maybe_unused]] const long long NP = op.N >> 1;       // pairs (bounds of the checked build)
    const int lane = threadIdx.x;
    const unsigned short* code2 = reinterpret_cast<const unsigned short*>(op.nbm);
    const unsigned short* lidx2 = reinterpret_cast<const unsigned short*>(op.lidx);
    const float2* x1 = reinterpret_cast<const float2*>(x);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    int l = i2 + h * (j + n * k0);
    float4 prev = z4, cur = z4, next = z4, fv = z4;
    if (NBR) {
        prev = (valid && k0 > 0) ? x[HCHK(l - sz, NP)] : z4;
        cur = valid ? x[HCHK(l, NP)] : z4;
        next = (valid && k0 + 1 < n) ? x[HCHK(l + sz, NP)] : z4;
    }
    if (RHS) fv = valid ? f[HCHK(l, NP)] : z4;
    unsigned cc = valid ? (unsigned)code2[HCHK(l, NP)] : kMM;
    unsigned li = valid ? (unsigned)lidx2[HCHK(l, NP)] : 0u;
    float acc = 0.f;
    float dre = 0.f, dim = 0.f, dtt = 0.f;                 // DOT sums
    float4 wv = z4;                                        // DOT operand, prefetched one plane ahead
    if (DOT) wv = valid ? dot.w[HCHK(l, NP)] : z4;
    for (int k = k0; k < k1; ++k, l += sz) {
        const bool more = valid && k + 1 < k1;
        float4 next2 = z4, f_n = z4, w_n = z4;
        if (DOT) w_n = more ? dot.w[HCHK(l + sz, NP)] : z4;
        if (NBR) next2 = (more && k + 2 < n) ? x[HCHK(l + 2 * sz, NP)] : z4;
        if (RHS) f_n = more ? f[HCHK(l + sz, NP)] : z4;
        const unsigned cc_n = more ? (unsigned)code2[HCHK(l + sz, NP)] : kMM;
        const unsigned li_n = more ? (unsigned)lidx2[HCHK(l + sz, NP)] : 0u;
        const unsigned c0 = cc & 0xffu, c1 = cc >> 8;
        float2 s0 = make_float2(0.f, 0.f), s1 = s0;
        if (NBR) {
            float2 left, right;
            left.x = __shfl_up_sync(0xffffffffu, cur.z, 1);
            left.y = __shfl_up_sync(0xffffffffu, cur.w, 1);
            right.x = __shfl_down_sync(0xffffffffu, cur.x, 1);
            right.y = __shfl_down_sync(0xffffffffu, cur.y, 1);
            // the row-segment ends: node i-1 of lane 0 and node i+2 of the last lane
            // (fluid nodes are interior, so these exist whenever the bit is set)
            if (lane == 0 && (c0 & 1u)) left = x1[HCHK(2 * l - 1, op.N)];
            if (lane == BX - 1 && (c1 & 2u)) right = x1[HCHK(2 * l + 2, op.N)];
            const unsigned any = c0 | c1;                  // a masked code has no neighbour bits
            const float4 ym = (any & 4u) ? x[HCHK(l - sy, NP)] : z4;
            const float4 yp = (any & 8u) ? x[HCHK(l + sy, NP)] : z4;
            pair_sums(c0, c1, left, right, cur, ym, yp, prev, next, s0, s1);
        }
        float2 o0, o1;
        if (KIND != 1) {
            float2 d0, d1;
            if (op.k2) {
                const float4 kk = reinterpret_cast<const float4*>(op.k2)[HCHK(l, NP)];
                d0 = make_float2(kk.x - 6.f * op.hinv2, kk.y);
                d1 = make_float2(kk.z - 6.f * op.hinv2, kk.w);
            } else {
                d0 = make_float2(op.dre, op.im[HCHK(li & 0xffu, kMaxLayerCells + 1)]);
                d1 = make_float2(op.dre, op.im[HCHK(li >> 8, kMaxLayerCells + 1)]);
            }
            if (conj) { d0.y = -d0.y; d1.y = -d1.y; }
            const float2 x0 = lo2(cur), xh = hi2(cur);
            o0 = (c0 & kMasked) ? x0
                                : make_float2(op.hinv2 * s0.x + (d0.x * x0.x - d0.y * x0.y),
                                              op.hinv2 * s0.y + (d0.x * x0.y + d0.y * x0.x));
            o1 = (c1 & kMasked) ? xh
                                : make_float2(op.hinv2 * s1.x + (d1.x * xh.x - d1.y * xh.y),
                                              op.hinv2 * s1.y + (d1.x * xh.y + d1.y * xh.x));
            if (FLAG || KIND == 2) {
                o0 = csub(lo2(fv), o0);
                o1 = csub(hi2(fv), o1);
            }
        } else {
            float2 id0, id1;
            if (op.k2) {
                const float4 iv = reinterpret_cast<const float4*>(op.invd)[HCHK(l, NP)];
                id0 = lo2(iv);
                id1 = hi2(iv);
            } else {
                id0 = op.invd_tab[HCHK(li & 0xffu, kMaxLayerCells + 1)];
                id1 = op.invd_tab[HCHK(li >> 8, kMaxLayerCells + 1)];
            }
            if (conj) { id0.y = -id0.y; id1.y = -id1.y; }
            const float2 f0 = lo2(fv), fh = hi2(fv);
            if (FLAG) {
                o0 = cscale(omega, (c0 & kMasked) ? f0 : cmul(id0, f0));
                o1 = cscale(omega, (c1 & kMasked) ? fh : cmul(id1, fh));
            } else {
                const float w1 = 1.f - omega;
                const float2 x0 = lo2(cur), xh = hi2(cur);
                if (c0 & kMasked) {
                    o0 = cadd(x0, cscale(omega, csub(f0, x0)));
                } else {
                    const float2 t = cmul(id0, make_float2(f0.x - op.hinv2 * s0.x, f0.y - op.hinv2 * s0.y));
                    o0 = make_float2(w1 * x0.x + omega * t.x, w1 * x0.y + omega * t.y);
                }
                if (c1 & kMasked) {
                    o1 = cadd(xh, cscale(omega, csub(fh, xh)));
                } else {
                    const float2 t = cmul(id1, make_float2(fh.x - op.hinv2 * s1.x, fh.y - op.hinv2 * s1.y));
                    o1 = make_float2(w1 * xh.x + omega * t.x, w1 * xh.y + omega * t.y);
                }
            }
        }
        if (valid && KIND == 2) {
            const int a = (j + k) & 1;                     // the red node of the pair
            const unsigned ca = a ? c1 : c0;
            reinterpret_cast<float2*>(y)[HCHK(l, NP)] = (ca & kMasked) ? make_float2(0.f, 0.f) : (a ? o1 : o0);
        } else if (valid) {
            y[HCHK(l, NP)] = make_float4(o0.x, o0.y, o1.x, o1.y);
            if (NORM) acc += (o0.x * o0.x + o0.y * o0.y) + (o1.x * o1.x + o1.y * o1.y);
            if (DOT == 1) {                                // conj(w) y
                const float2 w0 = lo2(wv), w1 = hi2(wv);
                dre = fmaf(w0.x, o0.x, fmaf(w0.y, o0.y, dre));
                dim = fmaf(w0.x, o0.y, fmaf(-w0.y, o0.x, dim));
                dre = fmaf(w1.x, o1.x, fmaf(w1.y, o1.y, dre));
                dim = fmaf(w1.x, o1.y, fmaf(-w1.y, o1.x, dim));
            } else if (DOT == 2) {                         // conj(y) w, |y|^2
                const float2 w0 = lo2(wv), w1 = hi2(wv);
                dre = fmaf(o0.x, w0.x, fmaf(o0.y, w0.y, dre));
                dim = fmaf(o0.x, w0.y, fmaf(-o0.y, w0.x, dim));
                dre = fmaf(o1.x, w1.x, fmaf(o1.y, w1.y, dre));
                dim = fmaf(o1.x, w1.y, fmaf(-o1.y, w1.x, dim));
                dtt = fmaf(o0.x, o0.x, fmaf(o0.y, o0.y, dtt));
                dtt = fmaf(o1.x, o1.x, fmaf(o1.y, o1.y, dtt));
            }
        }
        prev = cur;
        cur = next;
        next = next2;
        fv = f_n;
        wv = w_n;
        cc = cc_n;
        li = li_n;
    }
    if (NORM) {
        block_reduce_store<float>((double)acc, partials + (blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)));
        norm_tail(tail, partials, gridDim.x * gridDim.y * gridDim.z, threadIdx.x + BX * threadIdx.y);
    }
    if (DOT) {
        // S_STOP was set, if at all, by an earlier launch: every block takes the same
        // branch.  The block's partial sums only: the kernel that needs the scalar
        // (k32_s for alpha, k32_xr for omega) sums them itself.
        if (dot.sc[S_STOP].x != 0.0) return;
        // (FP32 butterflies and the warps in order: FP64 adds and shuffles run at a
        // small fraction of the FP32 rate on this GPU)
        constexpr int W = DOT == 1 ? 2 : 3;
        const int tid = threadIdx.x + BX * threadIdx.y;
        const unsigned bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
        float v[3] = {dre, dim, dtt};
        __shared__ float red[3][BX * BY / 32];
        for (int q = 0; q < W; ++q)
            for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
        if ((tid & 31) == 0)
            for (int q = 0; q < W; ++q) red[q][tid >> 5] = v[q];
        __syncthreads();
        if (tid < W) {
            float t = 0.f;
            for (int w = 0; w < BX * BY / 32; ++w) t += red[tid][w];
            dot.parts[W * bid + tid] = t;
        }
    }
}

// new value of a swept node (Gauss-Seidel, or SOR for omega != 1): a masked node
// takes f, a fluid node D^-1 (f - h^-2 s) from its neighbour sum s (D^-1 f when the
// old iterate is zero); SOR moves the old value xo by omega times the step
__device__ __forceinline__ float2 gs_value(const Op<float>& op, unsigned c, float2 fa, float2 s, float2 id,
                                           float2 xo, float omega, bool xzero) {
    float2 out;
    if (c & kMasked) {
        out = fa;
    } else if (xzero) {
        out = cmul(id, fa);
    } else {
        out = cmul(id, make_float2(fa.x - op.hinv2 * s.x, fa.y - op.hinv2 * s.y));
    }
    if (omega != 1.f) out = xzero ? cscale(omega, out) : cadd(xo, cscale(omega, csub(out, xo)));
    return out;
}

// complex64 red-black half-sweep in 3D with the pair layout of k_march_c64: each
// thread owns the node pair (2 i2, 2 i2 + 1) of a row, one node of each colour
// (n even), and updates the one of the swept colour in place.  The neighbours of
// that node are of the other colour and are not written by this launch, so the
// z-march keeps the planes in registers as in k_march_c64.  XZERO: the first
// half-sweep from x = 0 (no neighbours read).  SOR (omega != 1): the node moves by
// omega times its Gauss-Seidel step.
template <bool XZERO>
__global__ void __launch_bounds__(BX * BY) k_rbgs_c64(Op<float> op, int zc, int colour, const float4* __restrict__ f,
                                                      float4* x, int conj, float omega) {
    pdl_begin();
    constexpr unsigned kMM = kMasked | (kMasked << 8);
    const int n = op.n, h = n >> 1;
    const int i2 = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k0 = blockIdx.z * zc;
    const int k1 = min(n, k0 + zc);
    const bool valid = i2 < h && j < n;
    [[maybe_unused]] const long long NP = op.N >> 1;
    const int sy = h, sz = h * n;
    const int lane = threadIdx.x;
    const unsigned short* code2 = reinterpret_cast<const unsigned short*>(op.nbm);
    const unsigned short* lidx2 = reinterpret_cast<const unsigned short*>(op.lidx);
    const float2* x1 = reinterpret_cast<const float2*>(x);
    float2* xw = reinterpret_cast<float2*>(x);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    int l = i2 + h * (j + n * k0);
    float4 prev = z4, cur = z4, next = z4;
    if (!XZERO) {
        prev = (valid && k0 > 0) ? x[HCHK(l - sz, NP)] : z4;
        cur = valid ? x[HCHK(l, NP)] : z4;
        next = (valid && k0 + 1 < n) ? x[HCHK(l + sz, NP)] : z4;
    }
    float4 fv = valid ? f[HCHK(l, NP)] : z4;
    unsigned cc = valid ? (unsigned)code2[HCHK(l, NP)] : kMM;
    unsigned li = valid ? (unsigned)lidx2[HCHK(l, NP)] : 0u;
    for (int k = k0; k < k1; ++k, l += sz) {
        const bool more = valid && k + 1 < k1;
        float4 next2 = z4;
        if (!XZERO) next2 = (more && k + 2 < n) ? x[HCHK(l + 2 * sz, NP)] : z4;
        const float4 f_n = more ? f[HCHK(l + sz, NP)] : z4;
        const unsigned cc_n = more ? (unsigned)code2[HCHK(l + sz, NP)] : kMM;
        const unsigned li_n = more ? (unsigned)lidx2[HCHK(l + sz, NP)] : 0u;
        const int a = ((j + k) & 1) ^ colour;               // swept node of the pair
        const unsigned ca = a ? (cc >> 8) : (cc & 0xffu);
        float2 s0 = make_float2(0.f, 0.f), s1 = s0;
        if (!XZERO) {
            float2 left, right;
            left.x = __shfl_up_sync(0xffffffffu, cur.z, 1);
            left.y = __shfl_up_sync(0xffffffffu, cur.w, 1);
            right.x = __shfl_down_sync(0xffffffffu, cur.x, 1);
            right.y = __shfl_down_sync(0xffffffffu, cur.y, 1);
            if (lane == 0 && a == 0 && (ca & 1u)) left = x1[HCHK(2 * l - 1, op.N)];
            if (lane == BX - 1 && a == 1 && (ca & 2u)) right = x1[HCHK(2 * l + 2, op.N)];
            const float4 ym = (ca & 4u) ? x[HCHK(l - sy, NP)] : z4;
            const float4 yp = (ca & 8u) ? x[HCHK(l + sy, NP)] : z4;
            pair_sums(a ? 0u : ca, a ? ca : 0u, left, right, cur, ym, yp, prev, next, s0, s1);
        }
        if (valid) {
            float2 id = make_float2(0.f, 0.f);
            if (!(ca & kMasked)) {
                if (op.k2) {
                    const float4 iv = reinterpret_cast<const float4*>(op.invd)[HCHK(l, NP)];
                    id = a ? hi2(iv) : lo2(iv);
                } else {
                    id = op.invd_tab[HCHK(a ? (li >> 8) : (li & 0xffu), kMaxLayerCells + 1)];
                }
                if (conj) id.y = -id.y;
            }
            const float2 out = gs_value(op, ca, a ? hi2(fv) : lo2(fv), a ? s1 : s0, id, a ? hi2(cur) : lo2(cur),
                                        omega, XZERO);
            xw[HCHK(2 * l + a, op.N)] = out;
        }
        prev = cur;
        cur = next;
        next = next2;
        fv = f_n;
        cc = cc_n;
        li = li_n;
    }
}

// ---- one full red-black sweep per launch (complex64, 3D, n even, pair layout)
//
// Colour A (c0) on every node, then colour B (1 - c0), read from xin and written to xout
// (out of place).  A block owns whole x-rows: blockDim.x threads over the n/2 pairs of a
// row (a multiple of 32), blockDim.y = BYI + 2 rows, of which the first and last are halo
// rows: they compute the colour-A values of the rows just outside the block, which the
// block's own colour-B nodes need, instead of waiting for the neighbouring block.  Each
// thread marches in z over its pair; blocks split z into chunks and recompute the
// colour-A planes just outside their chunk.
//
// The kernel is bound by instruction issue before it is bound by HBM, so everything is
// kept split by colour rather than by position in the pair: which of a pair's two nodes is
// colour A alternates with row and plane, and only the loads of f and the tables and the
// store of the result swap by it.  All six neighbours of a node have the other colour, so
//  - only the colour-B half of xin is ever a neighbour: it is staged in shared memory, 8
//    bytes a pair, by asynchronous copies issued three planes ahead (a ring of four planes
//    of the block's rows plus one more row on each side);
//  - new colour-A values go to a ring of three shared planes; after one barrier the thread
//    updates colour B one plane behind;
//  - in both, one x-neighbour is the thread's own pair, the other the pair to the left or
//    right (alternating with the plane), y-neighbours are one row away, z-neighbours are
//    the thread's own values of the planes before and after.
// Old values of the swept nodes themselves are read only for SOR; without it the next sweep
// in the same order needs the colour-B nodes alone, so sweeps in a row pass just those on
// (CIN, COUT: xin, xout hold one float2 per pair; 18 B a node of reads and writes between
// two others, 22 at the ends of a run, instead of 26).  A node with all six
// neighbours fluid (the common case) takes no selects.  Every node value comes from the
// arithmetic of k_rbgs_c64 with the neighbour sums in the same order, so one launch equals
// two half-sweeps.  The roundings are spelled out (sor_step, cmul_n; cmul_t for colour A
// from zero), the same in every instantiation: left to the compiler they moved from one to
// the next by 2e-8, which the trunk-basis correction and eight FGMRES steps can raise to
// 1e-5 of the solution.  (f - h^-2 s can be fused in one way only; as fmaf it cost 2% of
// the sweep.)  Measured against the form that staged whole pairs and selected by
// position (431 instructions a pair at 256^3; ncu, cold): 256^3 133 -> 83 us a sweep (5.3
// TB/s of the 26 B a node), 128^3 20.5 -> 15.2 us, 64^3 13.2 -> 6.3 us.  The launch shape
// is chosen by plan_sweep32.

// neighbour sum of the node at position a of its pair: own, the pair's other node; side, the
// node across the pair's end (code bits select the fluid ones); the order of pair_sums
__device__ __forceinline__ float2 six_sum(unsigned c, int a, float2 own, float2 side, float2 ym, float2 yp, float2 zm,
                                          float2 zp) {
    if ((c & 0x3Fu) != 0x3Fu) {
        own = pick(c, a ? 1u : 2u, own);
        side = pick(c, a ? 2u : 1u, side);
        ym = pick(c, 4u, ym);
        yp = pick(c, 8u, yp);
        zm = pick(c, 16u, zm);
        zp = pick(c, 32u, zp);
    }
    return cadd(cadd(cadd(own, side), cadd(ym, yp)), cadd(zm, zp));
}

// x + omega (v - x)
__device__ __forceinline__ float2 sor_step(float2 x, float2 v, float omega) {
    return make_float2(fmaf(omega, v.x - x.x, x.x), fmaf(omega, v.y - x.y, x.y));
}

// 8-byte asynchronous copy global -> shared; valid = false fills zeros without reading
// (src must still be a mapped address)
__device__ __forceinline__ void cp_async8(void* dst, const void* src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// wait until at most N of this thread's copy groups are still in flight
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

constexpr int kSweepMaxThreads = 1024;
constexpr int kSweepXPlanes = 4;     // staged planes: t, t + 1, and two in flight

// dynamic shared memory of k_sweep_c64 for a block of txt x tyt threads
__host__ __device__ constexpr size_t sweep_smem_bytes(int txt, int tyt, bool xzero) {
    return ((xzero ? 0 : (size_t)kSweepXPlanes * (tyt + 2) * txt) + (size_t)3 * tyt * txt + kMaxLayerCells + 1) *
           sizeof(float2);
}

template <bool XZERO, bool SOR, bool K2, bool CIN, bool COUT>
__global__ void __launch_bounds__(kSweepMaxThreads, 1)
    k_sweep_c64(Op<float> op, int zc, int c0, const float4* __restrict__ f, const float2* __restrict__ xin,
                float2* __restrict__ xout, int conj, float omega) {
    pdl_begin();
    static_assert(!(SOR && (CIN || COUT)) && !(XZERO && CIN), "SOR reads the old values of both colours");
    extern __shared__ __align__(16) float2 sweep_smem[];
    constexpr unsigned kOut = kMasked | (kMasked << 16);   // (code, layer) byte pairs of two masked nodes
    const int n = op.n, h = n >> 1;
    const int TXT = blockDim.x, TYT = blockDim.y, BYI = TYT - 2;
    const int i2 = threadIdx.x, ty = threadIdx.y;
    const int j0 = blockIdx.y * BYI;                       // first inner row of the block
    const int j = j0 - 1 + ty;                             // this thread's row
    const int k0 = blockIdx.z * zc, k1 = min(n, k0 + zc);
    const bool row_ok = i2 < h && j >= 0 && j < n;
    const bool inner = row_ok && ty >= 1 && ty <= BYI;
    const int sz = h * n;
    [[maybe_unused]] const long long NP = op.N >> 1;
    const int RS = TYT + 2;                                // staged rows j0 - 2 .. j0 + BYI + 1
    const int PX = RS * TXT, PR = TYT * TXT;
    float2* xs = sweep_smem;                               // [4][RS][TXT] old colour-B values (not with XZERO)
    float2* ring = sweep_smem + (XZERO ? 0 : kSweepXPlanes * PX);   // [3][TYT][TXT] new colour-A values
    float2* stab = ring + 3 * PR;                          // 1/diag by layer index
    const int me = ty * TXT + i2;                          // this thread in a ring plane
    const int mx = me + TXT;                               // this thread's row in a staged plane
    const unsigned* cl2 = reinterpret_cast<const unsigned*>(op.ncl);
    const float2 z2 = make_float2(0.f, 0.f);
    const int lrow = i2 + h * j;
    if (!K2)
        for (int q = me; q <= op.L && q <= kMaxLayerCells; q += PR) {
            float2 v = op.invd_tab[q];
            if (conj) v.y = -v.y;
            stab[q] = v;
        }
    int t = k0 - 1;
    int ar = c0 ^ ((j + t) & 1);                           // position of the colour-A node at plane t
    // staged rows of this thread: its own, and the outer row next to a halo row
    const int jx = ty == 0 ? j0 - 2 : j0 + BYI + 1;
    const bool halo = !XZERO && (ty == 0 || ty == TYT - 1);
    const bool out_ok = halo && i2 < h && jx >= 0 && jx < n;
    const int mo = (ty == 0 ? 0 : RS - 1) * TXT + i2;
    const int lout = i2 + h * jx;
    // stage plane p (zeros outside the grid) at offset so; a: position of colour A there
    auto stage = [&](int p, int so, int a) {
        const bool pin = p >= 0 && p < n;
        auto at = [&](int q, int pos) { return CIN ? q : 2 * q + pos; };
        cp_async8(xs + so + mx, xin + HCHK(pin && row_ok ? at(lrow + sz * p, a ^ 1) : 0, CIN ? NP : op.N), pin && row_ok);
        if (halo) cp_async8(xs + so + mo, xin + HCHK(pin && out_ok ? at(lout + sz * p, a) : 0, CIN ? NP : op.N), pin && out_ok);
    };
    int o_0 = 0, o_p1 = PX, o_p2 = 2 * PX, o_p3 = 3 * PX;
    if (!XZERO) {
        stage(t, o_0, ar);
        stage(t + 1, o_p1, ar ^ 1);
        cp_async_commit();
        stage(t + 2, o_p2, ar);
        cp_async_commit();
        cp_async_wait<1>();
    }
    // this plane's f, tables, 1/diag (K2) and old colour-A value (SOR), by position
    const bool in0 = row_ok && t >= 0;
    float4 fc = make_float4(0.f, 0.f, 0.f, 0.f), ic = fc;
    unsigned cl = kOut;
    float2 xa = z2;
    if (in0) {
        const int l = lrow + sz * t;
        fc = f[HCHK(l, NP)];
        cl = cl2[HCHK(l, NP)];
        if (K2) ic = reinterpret_cast<const float4*>(op.invd)[HCHK(l, NP)];
        if (SOR && !XZERO) xa = xin[HCHK(2 * l + ar, op.N)];
    }
    // the pair to the left / right of this one (itself at the ends of the row: those nodes
    // lie on the masked ring and have no such neighbour)
    const int dl = i2 > 0 ? -1 : 0, dr = i2 + 1 < TXT ? 1 : 0;
    float2 am2 = z2, am1 = z2;                             // new colour-A values at planes t - 2, t - 1
    float2 fb = z2, xb = z2, ib = z2;                      // colour B of plane t - 1: f, old value, 1/diag
    unsigned cb = kMasked;                                 // its code and layer bytes
    float2 bm1 = z2, b0 = z2;                              // own old colour-B values at planes t - 1, t
    if (!XZERO && row_ok && t >= 1) {
        const int q = lrow + sz * (t - 1);
        bm1 = xin[HCHK(CIN ? q : 2 * q + ar, CIN ? NP : op.N)];
    }
    __syncthreads();
    if (!XZERO) b0 = xs[o_0 + mx];
    int rs = 0, rs_m = 2 * PR;                             // ring planes of t and t - 1
    int l = lrow + sz * t;
#pragma unroll 2
    for (; t <= k1; ++t, l += sz, ar ^= 1) {
        float4 fn = make_float4(0.f, 0.f, 0.f, 0.f), in = fn;
        unsigned cn = kOut;
        float2 xan = z2;
        if (row_ok && t + 1 < n) {
            fn = f[HCHK(l + sz, NP)];
            cn = cl2[HCHK(l + sz, NP)];
            if (K2) in = reinterpret_cast<const float4*>(op.invd)[HCHK(l + sz, NP)];
            if (SOR && !XZERO) xan = xin[HCHK(2 * (l + sz) + (ar ^ 1), op.N)];
        }
        const int dx = ar ? dr : dl;
        // colour A at plane t
        const float2 fa = ar ? hi2(fc) : lo2(fc);
        const unsigned ca = (ar ? cl >> 16 : cl) & 0xffffu;
        float2 bp1 = z2;
        if (!XZERO) bp1 = xs[o_p1 + mx];
        float2 na;
        if ((ca & 0xffu) == kMasked) {
            na = fa;
        } else {
            float2 id;
            if (K2) {
                id = ar ? hi2(ic) : lo2(ic);
                if (conj) id.y = -id.y;
            } else {
                id = stab[HCHK(ca >> 8, kMaxLayerCells + 1)];
            }
            if (XZERO) {
                na = cmul_t(id, fa);
            } else {
                const float2* P = xs + o_0 + mx;
                const float2 bx = P[dx];
                const float2 s = six_sum(ca, ar, b0, bx, P[-TXT], P[TXT], bm1, bp1);
                na = cmul_n(id, make_float2(fa.x - op.hinv2 * s.x, fa.y - op.hinv2 * s.y));
            }
        }
        if (SOR) na = XZERO ? cscale(omega, na) : sor_step(xa, na, omega);
        ring[rs + me] = na;
        if (!XZERO) {
            // plane t + 3 into the slot of plane t - 1 (last read before the previous step's
            // barrier); plane t + 2 (issued one step ago) must have landed before this one
            stage(t + 3, o_p3, ar ^ 1);
            cp_async_commit();
            cp_async_wait<1>();
        }
        __syncthreads();
        // colour B at plane t - 1 (its position there is that of colour A at plane t)
        if (inner && t - 1 >= k0 && t - 1 < k1) {
            float2 nb;
            if ((cb & 0xffu) == kMasked) {
                nb = fb;
            } else {
                const float2* R = ring + rs_m + me;
                const float2 ax = R[dx];
                const float2 s = six_sum(cb, ar, am1, ax, R[-TXT], R[TXT], am2, na);
                float2 id = ib;
                if (!K2) id = stab[HCHK(cb >> 8, kMaxLayerCells + 1)];
                else if (conj) id.y = -id.y;
                nb = cmul_n(id, make_float2(fb.x - op.hinv2 * s.x, fb.y - op.hinv2 * s.y));
            }
            // (from zero only colour A starts from zero: colour B's own old value is zero too)
            if (SOR) nb = sor_step(xb, nb, omega);
            if (COUT)
                xout[HCHK(l - sz, NP)] = nb;
            else
                reinterpret_cast<float4*>(xout)[HCHK(l - sz, NP)] =
                    ar ? make_float4(am1.x, am1.y, nb.x, nb.y) : make_float4(nb.x, nb.y, am1.x, am1.y);
        }
        am2 = am1;
        am1 = na;
        // the colour-B node at plane t is swept next step
        fb = ar ? lo2(fc) : hi2(fc);
        cb = (ar ? cl : cl >> 16) & 0xffffu;
        if (K2) ib = ar ? lo2(ic) : hi2(ic);
        if (SOR) xb = b0;
        bm1 = b0;
        b0 = bp1;
        fc = fn;
        cl = cn;
        if (K2) ic = in;
        if (SOR) xa = xan;
        rs_m = rs;
        rs = rs == 2 * PR ? 0 : rs + PR;
        const int o_free = o_0;
        o_0 = o_p1;
        o_p1 = o_p2;
        o_p2 = o_p3;
        o_p3 = o_free;
    }
    if (!XZERO) cp_async_wait<0>();
}

// y = A x, or y = f - A x (resid); two z-planes per thread; optional per-block ||y||^2 partials.
template <typename R, bool RESID, bool NORM>
__global__ void __launch_bounds__(BX * BY) k_apply(Op<R> op, int zc, const typename CT<R>::T* __restrict__ x,
                                                   const typename CT<R>::T* __restrict__ f,
                                                   typename CT<R>::T* __restrict__ y, double* partials,
                                                   int conj, NormTail tail) {
    pdl_begin();
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    // 3D: zc planes per block (noalloc_grid_blocks counts this grid's blocks)
    const int k0 = op.dim == 3 ? zc * blockIdx.z : 0;
    const int k1 = op.dim == 3 ? min(op.n, k0 + zc) : 1;
    double acc = 0.0;
    if (i < op.n && j < op.n)
        for (int kk = k0; kk < k1; ++kk)
            acc = norm_acc(apply_point<R, RESID>(op, x, f, y, conj, i, j, kk, i + (long long)op.n * (j + (long long)op.n * kk)),
                           acc);
    if (NORM) {
        block_reduce_store<R>(acc, partials + (blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)));
        norm_tail(tail, partials, gridDim.x * gridDim.y * gridDim.z, threadIdx.x + BX * threadIdx.y);
    }
}

// the end of a BiCGStab operator kernel: the block's sums a (and c) into parts, and in the
// last block the scalar update
template <int MODE>
__device__ __forceinline__ void bicg_finish(double2 a, double c, int tid, double2* sc, double* parts, unsigned* counter) {
    constexpr int W = MODE == 1 ? 2 : 3;
    double v[3] = {a.x, a.y, c};
    block_tree<W>(v, tid);
    if (tid == 0)
        for (int q = 0; q < W; ++q) parts[W * blockIdx.x + q] = v[q];
    if (last_block_done(counter, gridDim.x)) {
        sum_parts<W>(parts, gridDim.x, tid, v);
        if (tid == 0) {
            if (MODE == 1) bicg_alpha(sc, make_double2(v[0], v[1]));
            else bicg_omega(sc, make_double2(v[0], v[1]), v[2]);
            *counter = 0;
        }
    }
}

// y = A x with a BiCGStab reduction in the epilogue and its scalar update in the
// last block.  mode 1: <w, y> -> alpha = rho / <rhat, v> (w = rhat);
// mode 2: <y, w>, <y, y> -> omega (w = s).  Two nodes per thread, 512 consecutive ones
// per block (every lane busy whatever the row length).
constexpr int BN = 2;                 // nodes per thread
template <int MODE>
__global__ void __launch_bounds__(kFusedThreads) k_apply_bicg(Op<double> op, const double2* __restrict__ x,
                                                              double2* __restrict__ y, const double2* __restrict__ w,
                                                              int conj, double2* sc, double* parts, unsigned* counter) {
    pdl_begin();
    double2 a = make_double2(0, 0);
    double c = 0;
#pragma unroll
    for (int u = 0; u < BN; ++u) {
        const long long l = (blockIdx.x * (long long)BN + u) * kFusedThreads + threadIdx.x;
        if (l >= op.N) break;
        const double2 yv = apply_point<double, false>(op, x, nullptr, y, conj, 0, 0, 0, l), wv = w[l];
        a = MODE == 1 ? cfmac(wv, yv, a) : cfmac(yv, wv, a);
        if (MODE == 2) c = cnorm2(yv, c);
    }
    bicg_finish<MODE>(a, c, threadIdx.x, sc, parts, counter);
}

// one damped-Jacobi sweep: xout = xin + omega D^-1 (f - A xin), evaluated on a
// fluid node as (1 - omega) x + omega D^-1 (f - h^-2 sum of fluid neighbours)
// (the diagonal term cancels: fewer FP64 operations, same value up to rounding)
template <typename R, bool XZERO>
__device__ __forceinline__ void jacobi_point(const Op<R>& op, R omega, const typename CT<R>::T* __restrict__ f,
                                             const typename CT<R>::T* __restrict__ xin,
                                             typename CT<R>::T* __restrict__ xout, int conj, long long l) {
    using C = typename CT<R>::T;
    const C fl = f[l];
    // (by node_code, although every handle has the table: the compiler orders the loads better
    // behind its test; read straight from the table 256^3 took 871 us, 1024^2 49.3 for 42.7)
    const unsigned code = node_code(op, l);
    C out;
    if (code & kMasked) {
        if (XZERO) {
            out = cscale(omega, fl);
        } else {
            const C xc = xin[l];
            out = cadd(xc, cscale(omega, csub(fl, xc)));
        }
    } else {
        C id = invd_of(op, l, op.lidx[l], conj);
        if (XZERO) {
            out = cscale(omega, cmul(id, fl));
        } else {
            const C xc = xin[l];
            const C s = nbr_sum(op, xin, l, code);
            C g;
            g.x = fl.x - op.hinv2 * s.x;
            g.y = fl.y - op.hinv2 * s.y;
            const C t = cmul(id, g);
            const R w1 = (R)1 - omega;
            out.x = w1 * xc.x + omega * t.x;
            out.y = w1 * xc.y + omega * t.y;
        }
    }
    xout[l] = out;
}

// One node per thread in the flat order: every lane has a node whatever the row length
// (as in k_apply_z and the red-black kernels below).  In complex128, 32 x 8 tiles with two
// planes a thread and this: 97^3 59.5 and 51.4 us, 128^3 108.8 and 104.9, 256^3 785 and 783.
template <typename R, bool XZERO>
__global__ void __launch_bounds__(BX * BY) k_jacobi(Op<R> op, R omega, const typename CT<R>::T* __restrict__ f,
                                                    const typename CT<R>::T* __restrict__ xin,
                                                    typename CT<R>::T* __restrict__ xout, int conj) {
    pdl_begin();
    const long long l = blockIdx.x * (long long)(BX * BY) + threadIdx.x;
    if (l < op.N) jacobi_point<R, XZERO>(op, omega, f, xin, xout, conj, l);
}

// Several damped-Jacobi sweeps of a 2D grid in one launch (small grids, where a sweep
// costs its launch: 3 us at 64 x 64 against 0.1 us of FP64 arithmetic).  A block owns
// TI x TI nodes and recomputes a halo of S nodes around them, one node per thread
// (blockDim = TI + 2 S per side): S sweeps run in shared memory, each on a region one
// node smaller per side, and only the block's own nodes are written.  In FP64 the sweep is
// x <- (1 - omega) x + omega D^-1 f - omega h^-2 D^-1 s with the two products of D^-1
// formed once per node (12 FP64 instructions a sweep against 16 when D^-1 (f - h^-2 s)
// is formed each time).  In FP32, where instructions are cheap and a cycle's last bits show
// in the fifth digit of a mixed-precision solution, it is jacobi_point's formula with the
// same roundings, so that the tiled sweeps equal single ones bit for bit.  A masked node is
// zero to its neighbours.  xin = nullptr: from zero.
template <typename R>
__global__ void k_jacobi_tile(Op<R> op, R omega, int S, const typename CT<R>::T* __restrict__ f,
                              const typename CT<R>::T* __restrict__ xin, typename CT<R>::T* __restrict__ xout,
                              int conj) {
    pdl_begin();
    using C = typename CT<R>::T;
    constexpr bool kSplit = std::is_same<R, double>::value;
    extern __shared__ __align__(16) unsigned char jt_smem[];
    const int E = blockDim.x, TI = E - 2 * S, tx = threadIdx.x, ty = threadIdx.y, t = ty * E + tx;
    C* buf = reinterpret_cast<C*>(jt_smem);                // [2][E * E]
    const int i = blockIdx.x * TI - S + tx, j = blockIdx.y * TI - S + ty;
    const bool in = i >= 0 && j >= 0 && i < op.n && j < op.n;
    const int l = in ? i + op.n * j : 0;
    C zero;
    zero.x = 0; zero.y = 0;
    C x = zero, fp = zero, c = zero;
    bool fluid = false;
    if (in) {
        fluid = !(op.nbm[HCHK(l, op.N)] & kMasked);
        const C fv = f[HCHK(l, op.N)];
        if (xin) x = xin[HCHK(l, op.N)];
        if (kSplit) {                                      // fp: omega D^-1 f, c: omega h^-2 D^-1
            if (fluid) {
                const C id = cscale(omega, invd_of(op, l, op.lidx[HCHK(l, op.N)], conj));
                fp = cmul(id, fv);
                c = cscale(op.hinv2, id);
            } else {
                fp = cscale(omega, fv);
            }
        } else {                                           // fp: f, c: D^-1
            fp = fv;
            if (fluid) c = invd_of(op, l, op.lidx[HCHK(l, op.N)], conj);
        }
    }
    const int rim = min(min(tx, E - 1 - tx), min(ty, E - 1 - ty));
    const R w1 = (R)1 - omega;
    for (int q = 0; q < S; ++q) {
        C* b = buf + (q & 1) * E * E;
        b[t] = fluid ? x : zero;
        __syncthreads();
        if (rim > q) {
            C s = zero;
            if (fluid) s = cadd(cadd(b[t - 1], b[t + 1]), cadd(b[t - E], b[t + E]));
            if constexpr (kSplit) {
                C y;
                y.x = fp.x + w1 * x.x;
                y.y = fp.y + w1 * x.y;
                if (fluid) {
                    y.x -= c.x * s.x - c.y * s.y;
                    y.y -= c.x * s.y + c.y * s.x;
                }
                x = y;
            } else if (fluid) {
                const C d = cmul_n(c, make_float2(fmaf(-op.hinv2, s.x, fp.x), fmaf(-op.hinv2, s.y, fp.y)));
                x = make_float2(fmaf(w1, x.x, __fmul_rn(omega, d.x)), fmaf(w1, x.y, __fmul_rn(omega, d.y)));
            } else {
                x = sor_step(x, fp, omega);
            }
        }
    }
    if (rim >= S && in) xout[HCHK(l, op.N)] = x;
}

// red-black Gauss-Seidel update of one node of the swept colour, in place:
// x_l = D_l^-1 (f_l - h^-2 sum of fluid neighbours) on fluid nodes (the Gauss-Seidel
// value x + D^-1 (f - A x) with the diagonal term cancelled), f_l on masked nodes;
// SOR (omega != 1): x_l + omega (that value - x_l)
template <typename R, bool XZERO>
__device__ __forceinline__ void rbgs_point(const Op<R>& op, const typename CT<R>::T* __restrict__ f,
                                           typename CT<R>::T* x, int conj, long long l, R omega, bool sor) {
    using C = typename CT<R>::T;
    const C fl = f[l];
    const unsigned code = op.nbm[l];
    C out;
    if (code & kMasked) {
        out = fl;
    } else {
        const C id = invd_of(op, l, op.lidx[l], conj);
        if (XZERO) {
            out = cmul(id, fl);
        } else {
            const C s = nbr_sum(op, x, l, code);
            C g;
            g.x = fl.x - op.hinv2 * s.x;
            g.y = fl.y - op.hinv2 * s.y;
            out = cmul(id, g);
        }
    }
    if (sor) {
        if (XZERO) {
            out = cscale(omega, out);
        } else {
            const C xo = x[l];
            out = cadd(xo, cscale(omega, csub(out, xo)));
        }
    }
    x[l] = out;
}

// colour of node l: (i + j + k) mod 2
__device__ __forceinline__ int colour_of(long long l, int n) {
    const unsigned ul = (unsigned)l, un = (unsigned)n;
    const unsigned r = ul / un;          // row index j + n k
    const unsigned kk = r / un;
    return (int)(((ul - r * un) + (r - kk * un) + kk) & 1u);
}

// One thread per node pair (2m, 2m + 1), which holds one node of each colour (rows of even
// length start on even l; for odd n the colour is the parity of l), in the flat order, so
// that every lane has a node: one row per warp left a quarter of the lanes of 96-node rows
// idle, and the kernel is bound by the FP64 pipe (16 instructions a node).  96^3: 24.2 ->
// 19.1 us a half-sweep (ncu, cold).
template <typename R, bool XZERO>
__global__ void __launch_bounds__(BX * BY) k_rbgs(Op<R> op, int colour, const typename CT<R>::T* __restrict__ f,
                                                  typename CT<R>::T* x, int conj, R omega, bool sor) {
    pdl_begin();
    const long long m2 = 2 * (blockIdx.x * (long long)(BX * BY) + threadIdx.x);
    if (m2 >= op.N) return;
    const long long l = m2 + (colour_of(m2, op.n) != colour);
    if (l < op.N) rbgs_point<R, XZERO>(op, f, x, conj, l, omega, sor);
}

// r_red[m] = (v - A z) at the red node of pair (2m, 2m + 1)
__global__ void __launch_bounds__(BX * BY) k_residual_red(Op<double> op, const double2* __restrict__ z,
                                                          const double2* __restrict__ v,
                                                          double2* __restrict__ r_red, int conj) {
    pdl_begin();
    const long long m = blockIdx.x * (long long)(BX * BY) + threadIdx.x;
    if (2 * m >= op.N) return;
    const long long l = 2 * m + colour_of(2 * m, op.n);
    if (l >= op.N) return;
    const double2 xc = z[l];
    const unsigned code = op.nbm[l];
    double2 out;
    if (code & kMasked) {
        out = xc;
    } else {
        const double2 s = nbr_sum(op, z, l, code);
        const double2 d = diag_of(op, l, op.lidx[l], conj);
        out.x = op.hinv2 * s.x + (d.x * xc.x - d.y * xc.y);
        out.y = op.hinv2 * s.y + (d.x * xc.y + d.y * xc.x);
    }
    r_red[m] = csub(v[l], out);
}

// ---- double-float red-black Gauss-Seidel for FP64 handles.  The sweeps of the
// hybrid cycle keep f and x as FP32 pairs (value = hi + lo, a 48-bit significand)
// and run on the FP32 pipes, which this GPU has ~64x more of than FP64 pipes:
// f is split once (the first red half-sweep), the residual leaves as pairs for the
// projection, and the prolongation converts back to FP64 once.  Additions are
// two-sums with one renormalisation, products an FMA-exact product plus the cross
// terms (the lo*lo term, ~2^-48 relative, is dropped).
__device__ __forceinline__ float2 df_norm(float s, float e) {
    const float h = s + e;
    return make_float2(h, e - (h - s));
}
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
    const float s = a.x + b.x;
    const float bb = s - a.x;
    float e = (a.x - (s - bb)) + (b.x - bb);
    e += a.y + b.y;
    return df_norm(s, e);
}
__device__ __forceinline__ float2 df_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
    const float p = a.x * b.x;
    float e = fmaf(a.x, b.x, -p);
    e = fmaf(a.x, b.y, e);
    e = fmaf(a.y, b.x, e);
    return df_norm(p, e);
}
__device__ __forceinline__ float2 df_split(double v) { return f64_to_pair(v); }

struct Cdf {          // complex double-float
    float2 re, im;
};
__device__ __forceinline__ Cdf cdf_load(const float4* p, long long l) {
    const float4 v = p[l];
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ float4 cdf_pack(Cdf a) { return make_float4(a.re.x, a.re.y, a.im.x, a.im.y); }
__device__ __forceinline__ Cdf cdf_add(Cdf a, Cdf b) { return {df_add(a.re, b.re), df_add(a.im, b.im)}; }
__device__ __forceinline__ Cdf cdf_sub(Cdf a, Cdf b) { return {df_add(a.re, df_neg(b.re)), df_add(a.im, df_neg(b.im))}; }
__device__ __forceinline__ Cdf cdf_scale(float2 s, Cdf a) { return {df_mul(s, a.re), df_mul(s, a.im)}; }
__device__ __forceinline__ Cdf cdf_mul(Cdf a, Cdf b) {
    return {df_add(df_mul(a.re, b.re), df_neg(df_mul(a.im, b.im))), df_add(df_mul(a.re, b.im), df_mul(a.im, b.re))};
}
__device__ __forceinline__ Cdf cdf_zero() { return {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
__device__ __forceinline__ Cdf invd_df(const DfTab& t, int m, int conj) {
    const float4 v = t.invd[m];
    Cdf d = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
    if (conj) d.im = df_neg(d.im);
    return d;
}

// sum of the fluid neighbours (same tree as nbr_sum)
__device__ __forceinline__ Cdf nbr_sum_df(const Op<double>& op, const float4* __restrict__ x, long long l,
                                          unsigned code) {
    const long long sy = op.n, sz = (long long)op.n * op.n;
    const Cdf a = (code & 1u) ? cdf_load(x, HCHK(l - 1, op.N)) : cdf_zero();
    const Cdf b = (code & 2u) ? cdf_load(x, HCHK(l + 1, op.N)) : cdf_zero();
    const Cdf c = (code & 4u) ? cdf_load(x, HCHK(l - sy, op.N)) : cdf_zero();
    const Cdf d = (code & 8u) ? cdf_load(x, HCHK(l + sy, op.N)) : cdf_zero();
    Cdf s = cdf_add(cdf_add(a, b), cdf_add(c, d));
    if (op.dim == 3) {
        const Cdf e = (code & 16u) ? cdf_load(x, HCHK(l - sz, op.N)) : cdf_zero();
        const Cdf f = (code & 32u) ? cdf_load(x, HCHK(l + sz, op.N)) : cdf_zero();
        s = cdf_add(s, cdf_add(e, f));
    }
    return s;
}

// fs = f as pairs on every node; x = D^-1 f on red fluid nodes, f on red masked
// nodes, 0 on black nodes (the first red half-sweep from x = 0)
__global__ void k_rbgs_df_first(Op<double> op, DfTab t, const double2* __restrict__ f, float4* __restrict__ fs,
                                float4* __restrict__ xs, int conj) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = op.dim == 3 ? blockIdx.z : 0;
    if (i >= op.n || j >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    const double2 fv = f[l];
    const Cdf F = {df_split(fv.x), df_split(fv.y)};
    fs[l] = cdf_pack(F);
    Cdf x = cdf_zero();
    if (((i + j + k) & 1) == 0) {
        const unsigned code = node_code(op, l);
        x = (code & kMasked) ? F : cdf_mul(invd_df(t, node_lidx(op, l, i, j, k), conj), F);
    }
    xs[l] = cdf_pack(x);
}

// one half-sweep of colour `colour`: x = D^-1 (f - h^-2 s) on fluid nodes, f on masked
__global__ void __launch_bounds__(BX * BY) k_rbgs_df(Op<double> op, DfTab t, int colour,
                                                     const float4* __restrict__ fs, float4* xs, int conj) {
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = op.dim == 3 ? blockIdx.z : 0;
    if (j >= op.n) return;
    const int i = 2 * (blockIdx.x * BX + threadIdx.x) + ((j + k + colour) & 1);
    if (i >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    const unsigned code = node_code(op, l);
    const Cdf F = cdf_load(fs, l);
    Cdf x;
    if (code & kMasked) {
        x = F;
    } else {
        const Cdf sum = nbr_sum_df(op, xs, l, code);
        x = cdf_mul(invd_df(t, node_lidx(op, l, i, j, k), conj), cdf_sub(F, cdf_scale(t.hinv2, sum)));
    }
    xs[l] = cdf_pack(x);
}

// r_red[l / 2] = (f - A x)_l on the red nodes, as pairs
__global__ void __launch_bounds__(BX * BY) k_residual_red_df(Op<double> op, DfTab t, const float4* __restrict__ fs,
                                                             const float4* __restrict__ xs,
                                                             float4* __restrict__ r_red, int conj) {
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = op.dim == 3 ? blockIdx.z : 0;
    if (j >= op.n) return;
    const int i = 2 * (blockIdx.x * BX + threadIdx.x) + ((j + k) & 1);
    if (i >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    const unsigned code = node_code(op, l);
    const Cdf x = cdf_load(xs, l);
    Cdf out;
    if (code & kMasked) {
        out = x;
    } else {
        const Cdf sum = nbr_sum_df(op, xs, l, code);
        const int m = node_lidx(op, l, i, j, k);
        const Cdf d = {t.dre, conj ? df_neg(t.im[m]) : t.im[m]};
        out = cdf_add(cdf_scale(t.hinv2, sum), cdf_mul(d, x));
    }
    r_red[l >> 1] = cdf_pack(cdf_sub(cdf_load(fs, l), out));
}

// y = A x with the BiCGStab reduction of k_apply_bicg, for an x given as FP32 pairs
// (the output of the double-float hybrid cycle): the operator in double-float on
// the FP32 pipes, y converted to FP64 once, the dots in FP64
// (or, IN32, for a complex64 x: exact pairs with lo = 0)
__device__ __forceinline__ Cdf cdf_load(const float2* p, long long l) {
    const float2 v = p[l];
    return {make_float2(v.x, 0.f), make_float2(v.y, 0.f)};
}

template <typename XT>
__device__ __forceinline__ Cdf nbr_sum_any(const Op<double>& op, const XT* __restrict__ x, long long l,
                                           unsigned code) {
    const long long sy = op.n, sz = (long long)op.n * op.n;
    const Cdf a = (code & 1u) ? cdf_load(x, HCHK(l - 1, op.N)) : cdf_zero();
    const Cdf b = (code & 2u) ? cdf_load(x, HCHK(l + 1, op.N)) : cdf_zero();
    const Cdf c = (code & 4u) ? cdf_load(x, HCHK(l - sy, op.N)) : cdf_zero();
    const Cdf d = (code & 8u) ? cdf_load(x, HCHK(l + sy, op.N)) : cdf_zero();
    Cdf s = cdf_add(cdf_add(a, b), cdf_add(c, d));
    if (op.dim == 3) {
        const Cdf e = (code & 16u) ? cdf_load(x, HCHK(l - sz, op.N)) : cdf_zero();
        const Cdf f = (code & 32u) ? cdf_load(x, HCHK(l + sz, op.N)) : cdf_zero();
        s = cdf_add(s, cdf_add(e, f));
    }
    return s;
}

template <int MODE, typename XT>
__global__ void __launch_bounds__(kFusedThreads) k_apply_bicg_df(Op<double> op, DfTab t, const XT* __restrict__ x,
                                                                 double2* __restrict__ y, const double2* __restrict__ w,
                                                                 int conj, double2* sc, double* parts,
                                                                 unsigned* counter) {
    pdl_begin();
    double2 a = make_double2(0, 0);
    double c = 0;
#pragma unroll
    for (int u = 0; u < BN; ++u) {
        const long long l = (blockIdx.x * (long long)BN + u) * kFusedThreads + threadIdx.x;
        if (l >= op.N) break;
        const unsigned code = op.nbm[l];
        const Cdf X = cdf_load(x, l);
        const double2 wv = w[l];
        Cdf out;
        if (code & kMasked) {
            out = X;
        } else {
            const Cdf sum = nbr_sum_any(op, x, l, code);
            const int m = op.lidx[l];
            const Cdf d = {t.dre, conj ? df_neg(t.im[m]) : t.im[m]};
            out = cdf_add(cdf_scale(t.hinv2, sum), cdf_mul(d, X));
        }
        const double2 yv = make_double2(pair_to_f64(out.re.x, out.re.y), pair_to_f64(out.im.x, out.im.y));
        y[l] = yv;
        a = MODE == 1 ? cfmac(wv, yv, a) : cfmac(yv, wv, a);
        if (MODE == 2) c = cnorm2(yv, c);
    }
    bicg_finish<MODE>(a, c, threadIdx.x, sc, parts, counter);
}

// ---- the red-black part of the trunk-basis hybrid cycle in one cooperative
// launch: f as pairs with the first red half-sweep from x = 0, the remaining
// half-sweeps, and the red-row residual, each phase over the whole grid and the
// phases separated by a grid barrier (one block per SM, all blocks resident).
// Values written in an earlier phase by other blocks are read past L1 (ld.cg).
// The barrier's wait is bounded: on a timeout it records *err and lets the block
// go on (the host reports the solve as failed).
struct GridBar {
    unsigned* count;        // arrivals in the current barrier
    unsigned* gen;          // barrier generation
    int* err;               // set to 1 when a wait gives up
    double2* sc;            // Krylov scalars or null: a timeout also stops the BiCGStab loop
    unsigned spin_limit;    // polls of the generation word before a wait gives up
    unsigned target;        // arrivals that complete a barrier (gridDim.x; more only to inject a timeout)
};

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// arrival is an acquire-release add on the counter (each block's writes, ordered
// before it by the block barrier, are released; the last arrival acquires them all),
// the last block resets the counter and releases the next generation, and the
// others acquire it.  Thread 0 waits for all; the block barrier passes it on.
__device__ __forceinline__ void grid_barrier(const GridBar& b) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned g = ld_acquire_gpu(b.gen);
        unsigned old;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(b.count) : "memory");
        if (old == b.target - 1) {
            asm volatile("st.relaxed.gpu.global.u32 [%0], 0;" ::"l"(b.count) : "memory");
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(b.gen) : "memory");
        } else {
            for (unsigned it = 0; ld_acquire_gpu(b.gen) == g; ++it)
                if (it >= b.spin_limit) {
                    // give up: record it and mark the BiCGStab iteration as stopped
                    // (flag 4 = timeout); the block goes on with its phases, reading
                    // and writing only in-range entries
                    atomicExch(b.err, 1);
                    if (b.sc) {
                        b.sc[S_FLAGS].y = 4.0;
                        b.sc[S_STOP].x = 1.0;
                    }
                    break;
                }
        }
    }
    __syncthreads();
}

__device__ __forceinline__ Cdf cdf_load_cg(const float4* p, long long l) {
    const float4 v = __ldcg(p + l);
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}

__device__ __forceinline__ Cdf nbr_sum_df_cg(const Op<double>& op, const float4* x, long long l, unsigned code) {
    const long long sy = op.n, sz = (long long)op.n * op.n;
    const Cdf a = (code & 1u) ? cdf_load_cg(x, HCHK(l - 1, op.N)) : cdf_zero();
    const Cdf b = (code & 2u) ? cdf_load_cg(x, HCHK(l + 1, op.N)) : cdf_zero();
    const Cdf c = (code & 4u) ? cdf_load_cg(x, HCHK(l - sy, op.N)) : cdf_zero();
    const Cdf d = (code & 8u) ? cdf_load_cg(x, HCHK(l + sy, op.N)) : cdf_zero();
    Cdf s = cdf_add(cdf_add(a, b), cdf_add(c, d));
    if (op.dim == 3) {
        const Cdf e = (code & 16u) ? cdf_load_cg(x, HCHK(l - sz, op.N)) : cdf_zero();
        const Cdf f = (code & 32u) ? cdf_load_cg(x, HCHK(l + sz, op.N)) : cdf_zero();
        s = cdf_add(s, cdf_add(e, f));
    }
    return s;
}

constexpr int kCycleThreads = 1024;

// PRE selects where the cycle's right-hand side comes from: 0, f as given; 1, the
// BiCGStab direction update p = r + beta (p - omega v) (p written back); 2, the
// BiCGStab half step s = r - alpha v (written to w) with ||s||^2 summed per block
// and, after the first barrier, in block 0 in a fixed order (scalar recurrence of
// the BiCGStab driver, slot S_SN2 and the tolerance flag)
template <int PRE>
__global__ void __launch_bounds__(kCycleThreads, 1) k_cycle_df(Op<double> op, DfTab t, const double2* __restrict__ f,
                                                               const double2* __restrict__ v, double2* w, double2* sc,
                                                               double* parts, double tol_abs, float4* fs, float4* xs,
                                                               float4* r_red, int n_r, int conj, GridBar bar) {
    const long long N = op.N, M = (N + 1) / 2;
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long nth = (long long)gridDim.x * blockDim.x;
    double2 c1 = make_double2(0, 0), c2 = c1;
    if (PRE == 1) { c1 = sc[S_BETA]; c2 = sc[S_OMEGA]; }
    if (PRE == 2) c1 = sc[S_ALPHA];
    double acc = 0.0;
    // fs = f as pairs; x = D^-1 f on red fluid nodes, f on red masked nodes, 0 on black
    for (long long l = tid; l < N; l += nth) {
        double2 fv;
        if (PRE == 0) {
            fv = f[l];
        } else if (PRE == 1) {
            fv = cfma(c1, cfma(make_double2(-c2.x, -c2.y), v[l], w[l]), f[l]);
            w[l] = fv;
        } else {
            fv = cfma(make_double2(-c1.x, -c1.y), v[l], f[l]);
            w[l] = fv;
            acc = cnorm2(fv, acc);
        }
        const Cdf F = {df_split(fv.x), df_split(fv.y)};
        __stcg(fs + l, cdf_pack(F));
        Cdf x = cdf_zero();
        if (colour_of(l, op.n) == 0) {
            const unsigned code = op.nbm[l];
            x = (code & kMasked) ? F : cdf_mul(invd_df(t, op.lidx[l], conj), F);
        }
        __stcg(xs + l, cdf_pack(x));
    }
    if (PRE == 2) {
        // fixed-order tree over the block (see block_tree for why not butterflies)
        __shared__ double red[kCycleThreads / 2];
        for (int h = kCycleThreads / 2; h >= 32; h >>= 1) {
            if ((int)threadIdx.x >= h && (int)threadIdx.x < 2 * h) red[threadIdx.x - h] = acc;
            __syncthreads();
            if ((int)threadIdx.x < h) acc += red[threadIdx.x];
            __syncthreads();
        }
        if (threadIdx.x < 32) {
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
            if (threadIdx.x == 0) parts[blockIdx.x] = acc;
        }
    }
    grid_barrier(bar);
    if (PRE == 2 && blockIdx.x == 0 && threadIdx.x < 32) {
        double sn = 0.0;
        for (unsigned b = threadIdx.x; b < gridDim.x; b += 32) sn += __ldcg(parts + b);
        for (int o = 16; o > 0; o >>= 1) sn += __shfl_down_sync(0xffffffffu, sn, o);
        if (threadIdx.x == 0) bicg_snorm(sc, sn, tol_abs);
    }
    for (int q = 0; q < n_r; ++q) {
        for (int colour = (q == 0 ? 1 : 0); colour < 2; ++colour) {
            for (long long m = tid; m < M; m += nth) {
                const long long l = 2 * m + (colour_of(2 * m, op.n) != colour);
                if (l >= N) continue;
                const unsigned code = op.nbm[l];
                const Cdf F = cdf_load_cg(fs, l);
                Cdf x;
                if (code & kMasked) {
                    x = F;
                } else {
                    const Cdf sum = nbr_sum_df_cg(op, xs, l, code);
                    x = cdf_mul(invd_df(t, op.lidx[l], conj), cdf_sub(F, cdf_scale(t.hinv2, sum)));
                }
                __stcg(xs + l, cdf_pack(x));
            }
            grid_barrier(bar);
        }
    }
    // r_red[m] = (f - A x) at the red node of pair m
    for (long long m = tid; m < M; m += nth) {
        const long long l = 2 * m + (colour_of(2 * m, op.n) != 0);
        const unsigned code = op.nbm[l];
        const Cdf x = cdf_load_cg(xs, l);
        Cdf out;
        if (code & kMasked) {
            out = x;
        } else {
            const Cdf sum = nbr_sum_df_cg(op, xs, l, code);
            const int mm = op.lidx[l];
            const Cdf d = {t.dre, conj ? df_neg(t.im[mm]) : t.im[mm]};
            out = cdf_add(cdf_scale(t.hinv2, sum), cdf_mul(d, x));
        }
        r_red[m] = cdf_pack(cdf_sub(cdf_load_cg(fs, l), out));
    }
}

__global__ void k_rhs(Op<double> op, const double2* __restrict__ src, const double2* __restrict__ g,
                      double2* __restrict__ b) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= op.n || j >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    if (op.mask[l]) {
        b[l] = g[l];
        return;
    }
    const long long sy = op.n, sz = (long long)op.n * op.n;
    double2 v = src[l];
    long long nb[6] = {l - 1, l + 1, l - sy, l + sy, l - sz, l + sz};
    const int nn = 2 * op.dim;
    for (int q = 0; q < nn; ++q) {
        if (op.mask[nb[q]]) {
            double2 gm = g[nb[q]];
            v.x -= gm.x * op.hinv2;
            v.y -= gm.y * op.hinv2;
        }
    }
    b[l] = v;
}

__global__ void k_layer_k2(Op<double> op, double k0sq, double strength, const double* __restrict__ scale,
                           double2* __restrict__ k2) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= op.n || j >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    const int m = node_layer(op, i, j, k);
    const double eta = op.L > 0 ? (double)m / (double)op.L : 0.0;
    const double base = scale ? k0sq * scale[l] : k0sq;
    k2[l] = make_double2(base, base * (strength * eta * eta));
}

__global__ void k_invd_field(Op<double> op, double2* __restrict__ invd) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= op.n || j >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    double2 d = op.k2[l];
    d.x -= 2.0 * op.dim * op.hinv2;
    invd[l] = op.mask[l] ? make_double2(1.0, 0.0) : cdiv(make_double2(1.0, 0.0), d);
}

__global__ void k_layer_index(Op<double> op, uint8_t* __restrict__ lidx) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= op.n || j >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    lidx[l] = (uint8_t)node_layer(op, i, j, k);
}

__global__ void k_nbr_code(Op<double> op, uint8_t* __restrict__ code) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= op.n || j >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    const long long sy = op.n, sz = (long long)op.n * op.n;
    unsigned c = 0;
    if (op.mask[l]) {
        c = kMasked;
    } else if (op.face) {
        // outer-boundary problem: a neighbour counts if it is in the grid and unmasked
        const int n = op.n;
        if (i > 0 && !op.mask[l - 1]) c |= 1u;
        if (i < n - 1 && !op.mask[l + 1]) c |= 2u;
        if (j > 0 && !op.mask[l - sy]) c |= 4u;
        if (j < n - 1 && !op.mask[l + sy]) c |= 8u;
        if (op.dim == 3) {
            if (k > 0 && !op.mask[l - sz]) c |= 16u;
            if (k < n - 1 && !op.mask[l + sz]) c |= 32u;
        }
    } else {
        // fluid nodes are interior (the outer ring is masked), so all neighbours exist
        if (!op.mask[l - 1]) c |= 1u;
        if (!op.mask[l + 1]) c |= 2u;
        if (!op.mask[l - sy]) c |= 4u;
        if (!op.mask[l + sy]) c |= 8u;
        if (op.dim == 3) {
            if (!op.mask[l - sz]) c |= 16u;
            if (!op.mask[l + sz]) c |= 32u;
        }
    }
    code[l] = (uint8_t)c;
}

// ncl[l] = neighbour code | layer index << 8: one load a pair for both tables
__global__ void k_node_pack(const uint8_t* __restrict__ code, const uint8_t* __restrict__ lidx,
                            uint16_t* __restrict__ ncl, long long N) {
    for (long long l = blockIdx.x * (long long)blockDim.x + threadIdx.x; l < N; l += (long long)gridDim.x * blockDim.x)
        ncl[l] = (uint16_t)(code[l] | (lidx[l] << 8));
}

// face byte of a node: (number of boundary faces << 4) | axis bits
__global__ void k_face_code(Op<double> op, uint8_t* __restrict__ face) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= op.n || j >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    const int n = op.n;
    const unsigned ax = (i == 0 || i == n - 1) ? 1u : 0u, ay = (j == 0 || j == n - 1) ? 1u : 0u;
    const unsigned az = (op.dim == 3 && (k == 0 || k == n - 1)) ? 1u : 0u;
    face[l] = (uint8_t)(((ax + ay + az) << 4) | ax | (ay << 1) | (az << 2));
}

// effective k^2 of the outer-boundary problem: with it diag_of returns the scaled
// boundary diagonal 2^-b (k^2 - 2d h^-2 + 2 i k0 a / h), a = number of Sommerfeld
// faces of the node (all its faces but the Neumann top face y = 1 in 2D, z = 1 in 3D)
__global__ void k_bvp_k2(Op<double> op, const double2* __restrict__ k2phys, double k0, int neumann_top,
                         double2* __restrict__ k2eff) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= op.n || j >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    const int n = op.n;
    const int top = op.dim == 3 ? (k == n - 1) : (j == n - 1);
    const int nb = (i == 0) + (i == n - 1) + (j == 0) + (j == n - 1) + (op.dim == 3 ? (k == 0) + (k == n - 1) : 0);
    const int a = nb - (neumann_top && top ? 1 : 0);
    const double sigma = ldexp(1.0, -nb), h = sqrt(1.0 / op.hinv2), two_d = 2.0 * op.dim * op.hinv2;
    const double2 kp = k2phys ? k2phys[l] : make_double2(k0 * k0, 0.0);
    // K - 2d h^-2 = sigma (k^2 - 2d h^-2) + i sigma 2 k0 a / h
    k2eff[l] = make_double2(sigma * (kp.x - two_d) + two_d, sigma * (kp.y + 2.0 * k0 * a / h));
}

// right-hand side of the outer-boundary problem: masked nodes carry the Dirichlet
// value g; a fluid node gets 2^-b (src - (2 / h) g [on the Neumann top face]) minus the
// weighted Dirichlet values of its masked neighbours
__global__ void k_rhs_bvp(Op<double> op, const double2* __restrict__ src, const double2* __restrict__ g,
                          int neumann_top, double2* __restrict__ b) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= op.n || j >= op.n) return;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    if (op.mask[l]) {
        b[l] = g[l];
        return;
    }
    const int n = op.n;
    const unsigned fc = op.face[l];
    const int nb = (int)(fc >> 4);
    const double sigma = ldexp(1.0, -nb), h = sqrt(1.0 / op.hinv2);
    const int top = op.dim == 3 ? (k == n - 1) : (j == n - 1);
    double2 v = src[l];
    if (neumann_top && top) {
        v.x -= 2.0 / h * g[l].x;
        v.y -= 2.0 / h * g[l].y;
    }
    v = cscale(sigma, v);
    const long long sy = n, sz = (long long)n * n;
    const double wx = ldexp(1.0, -(nb - (int)(fc & 1u))), wy = ldexp(1.0, -(nb - (int)((fc >> 1) & 1u)));
    const double wz = ldexp(1.0, -(nb - (int)((fc >> 2) & 1u)));
    auto lift = [&](bool exists, long long m, double w) {
        if (exists && op.mask[m]) {
            v.x -= op.hinv2 * w * g[m].x;
            v.y -= op.hinv2 * w * g[m].y;
        }
    };
    lift(i > 0, l - 1, wx);
    lift(i < n - 1, l + 1, wx);
    lift(j > 0, l - sy, wy);
    lift(j < n - 1, l + sy, wy);
    if (op.dim == 3) {
        lift(k > 0, l - sz, wz);
        lift(k < n - 1, l + sz, wz);
    }
    b[l] = v;
}

__global__ void k_check_ring(Op<double> op, int* bad) {
    const int i = blockIdx.x * BX + threadIdx.x;
    const int j = blockIdx.y * BY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= op.n || j >= op.n) return;
    bool ring = i == 0 || j == 0 || i == op.n - 1 || j == op.n - 1;
    if (op.dim == 3) ring = ring || k == 0 || k == op.n - 1;
    const long long l = i + (long long)op.n * (j + (long long)op.n * k);
    if (ring && !op.mask[l]) atomicOr(bad, 1);
}

dim3 grid_for(int dim, int n, int xdiv = 1, int zdiv = 1) {
    int nx = (n + xdiv - 1) / xdiv;
    return dim3((nx + BX - 1) / BX, (n + BY - 1) / BY, dim == 3 ? (n + zdiv - 1) / zdiv : 1);
}

}  // namespace

namespace {
long long node_count(int dim, int n) { return dim == 3 ? (long long)n * n * n : (long long)n * n; }
// blocks of BX * BY threads, one element each
unsigned flat_blocks(long long count) { return (unsigned)((count + BX * BY - 1) / (BX * BY)); }
}  // namespace

int bicg_grid_blocks(int dim, int n) {
    return (int)((node_count(dim, n) + BN * kFusedThreads - 1) / (BN * kFusedThreads));
}

constexpr int ZC = 16;      // largest z chunk

// z chunk of a 3D marching grid with xy blocks per plane: the largest of 16, 8,
// 4, 2, 1 that leaves at least four blocks per SM
int march_zc(long long xy, int n) {
    int zc = ZC;
    while (zc > 1 && xy * ((n + zc - 1) / zc) < 4 * 152) zc /= 2;
    return zc;
}

int apply_zc(int dim, int n) {
    if (dim != 3) return 1;
    return march_zc((long long)((n + BX - 1) / BX) * ((n + BY - 1) / BY), n);
}

// grid of k_apply_z: the z chunk of 2 to 8 planes for which the busiest SM walks the fewest
// planes (its share of the blocks, times their planes and, with a norm, half a plane for the
// sums of each), so that the blocks come out in whole rounds.  Not more than 8 planes: a
// longer chunk reads fewer planes twice but leaves an SM too few blocks to cover their
// loads, which the count of planes does not see.  Apply and residual in complex128, us,
// with one plane for the start of a block and no limit, and by this rule: 192^3 (192 planes,
// one block an SM) 307 and 400, 240 and 308; 256^3 (64 planes) 602 and 730, 556 and 705;
// 129^3 (15) 82 and 104, 75 and 99; 96^3 (24) 36 and 46, 32 and 44.
dim3 applyz_grid(int n, bool norm, int* zc) {
    const long long per = ((long long)n * n + AZ - 1) / AZ;
    long long best = 0;
    *zc = 1;
    for (int z = std::min(8, n); z >= std::min(2, n); --z) {
        const long long blocks = per * ((n + z - 1) / z), cost = (blocks + 151) / 152 * (2 * z + (norm ? 1 : 0));
        if (best == 0 || cost < best) {
            best = cost;
            *zc = z;
        }
    }
    return dim3((unsigned)per, (n + *zc - 1) / *zc);
}

// grid of the two-nodes-per-thread complex64 kernels
dim3 pair_grid(int n, int* zc) {
    const int h = n / 2;
    const int gx = (h + BX - 1) / BX, gy = (n + BY - 1) / BY;
    *zc = march_zc((long long)gx * gy, n);
    return dim3(gx, gy, (n + *zc - 1) / *zc);
}

bool aligned16(const void* p) { return p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// the complex64 pair kernels apply: 3D, tables present, n even, 16-byte aligned vectors
bool pair_ok(const Op<float>& op, const void* a, const void* b, const void* c) {
    return op.dim == 3 && op.nbm && op.lidx && !op.face && (op.n % 2) == 0 && aligned16(a) && aligned16(b) && aligned16(c) &&
           aligned16(op.k2) && aligned16(op.invd);
}

// blocks of the table-free operator (one partial sum each)
int noalloc_grid_blocks(int dim, int n) {
    dim3 g = grid_for(dim, n, 1, apply_zc(dim, n));
    long long b = (long long)g.x * g.y * g.z;
    if (dim == 3 && n % 2 == 0) {
        int zc;
        dim3 p = pair_grid(n, &zc);
        b = std::max(b, (long long)p.x * p.y * p.z);
    }
    return (int)b;
}

// an upper bound on the partial sums any operator launch writes (buffer sizing)
int apply_grid_blocks(int dim, int n) {
    long long b = noalloc_grid_blocks(dim, n);
    if (dim == 3) {
        int zc;
        const dim3 g = applyz_grid(n, true, &zc);
        b = std::max(b, (long long)g.x * g.y);
    }
    return (int)b;
}

template <typename R>
int launch_apply(const Op<R>& op, const typename CT<R>::T* x, const typename CT<R>::T* f, typename CT<R>::T* y,
                 double* partials, int conj, bool resid, cudaStream_t s, double* norm, unsigned* counters) {
    auto tail_of = [&](NormRoute r) { return NormTail{norm, counters ? counters + r : nullptr}; };
    if constexpr (std::is_same<R, float>::value) {
        if (pair_ok(op, x, resid ? f : nullptr, y)) {
            int zc;
            const dim3 g = pair_grid(op.n, &zc), b(BX, BY);
            const float4* x4 = reinterpret_cast<const float4*>(x);
            const float4* f4 = reinterpret_cast<const float4*>(f);
            float4* y4 = reinterpret_cast<float4*>(y);
            const NormTail tail = tail_of(kNormPairs);
            if (resid) {
                if (partials) launch_after(k_march_c64<0, true, true>, g, b, 0, s, op, zc, 0.f, x4, f4, y4, partials, conj, Dot32{}, tail);
                else launch_after(k_march_c64<0, true, false>, g, b, 0, s, op, zc, 0.f, x4, f4, y4, partials, conj, Dot32{}, tail);
            } else {
                if (partials) launch_after(k_march_c64<0, false, true>, g, b, 0, s, op, zc, 0.f, x4, f4, y4, partials, conj, Dot32{}, tail);
                else launch_after(k_march_c64<0, false, false>, g, b, 0, s, op, zc, 0.f, x4, f4, y4, partials, conj, Dot32{}, tail);
            }
            return (int)(g.x * g.y * g.z);
        }
    }
    if (op.dim == 3 && op.nbm && op.lidx && !op.face) {
        int zc;
        const dim3 g = applyz_grid(op.n, partials != nullptr, &zc);
        const NormTail tail = tail_of(kNormZ);
        if (resid) {
            if (partials) launch_after(k_apply_z<R, true, true>, g, AZ, 0, s, op, zc, x, f, y, partials, conj, tail);
            else launch_after(k_apply_z<R, true, false>, g, AZ, 0, s, op, zc, x, f, y, partials, conj, tail);
        } else {
            if (partials) launch_after(k_apply_z<R, false, true>, g, AZ, 0, s, op, zc, x, f, y, partials, conj, tail);
            else launch_after(k_apply_z<R, false, false>, g, AZ, 0, s, op, zc, x, f, y, partials, conj, tail);
        }
        return (int)(g.x * g.y);
    }
    const int zc = apply_zc(op.dim, op.n);
    dim3 g = grid_for(op.dim, op.n, 1, zc), b(BX, BY);
    // 2D, or an operator without the per-node tables (the allocation-free path)
    const NormTail tail = tail_of(kNormFlat);
    if (resid) {
        if (partials) launch_after(k_apply<R, true, true>, g, b, 0, s, op, zc, x, f, y, partials, conj, tail);
        else launch_after(k_apply<R, true, false>, g, b, 0, s, op, zc, x, f, y, partials, conj, tail);
    } else {
        if (partials) launch_after(k_apply<R, false, true>, g, b, 0, s, op, zc, x, f, y, partials, conj, tail);
        else launch_after(k_apply<R, false, false>, g, b, 0, s, op, zc, x, f, y, partials, conj, tail);
    }
    return (int)(g.x * g.y * g.z);
}

template <typename R>
void launch_jacobi(const Op<R>& op, double omega, const typename CT<R>::T* f, const typename CT<R>::T* xin,
                   typename CT<R>::T* xout, int conj, bool xzero, cudaStream_t s) {
    if constexpr (std::is_same<R, float>::value) {
        if (pair_ok(op, f, xzero ? nullptr : xin, xout)) {
            int zc;
            const dim3 g = pair_grid(op.n, &zc), b(BX, BY);
            const float4* x4 = reinterpret_cast<const float4*>(xin);
            const float4* f4 = reinterpret_cast<const float4*>(f);
            float4* y4 = reinterpret_cast<float4*>(xout);
            if (xzero) launch_after(k_march_c64<1, true, false>, g, b, 0, s, op, zc, (float)omega, x4, f4, y4, nullptr, conj, Dot32{}, NormTail{});
            else launch_after(k_march_c64<1, false, false>, g, b, 0, s, op, zc, (float)omega, x4, f4, y4, nullptr, conj, Dot32{}, NormTail{});
            return;
        }
    }
    const unsigned g = flat_blocks(op.N);
    if (xzero) launch_after(k_jacobi<R, true>, g, BX * BY, 0, s, op, (R)omega, f, xin, xout, conj);
    else launch_after(k_jacobi<R, false>, g, BX * BY, 0, s, op, (R)omega, f, xin, xout, conj);
}

// sweeps per launch of the tiled form for this operator, 0 where it does not apply (3D,
// outer-boundary rows, no tables) or does not pay: with the halo a node costs two to four
// times its arithmetic, so the tiles win while a sweep is bound by its launch.  20 sweeps,
// us, single ones and tiled: complex128 128^2 59.0 and 40.6, 192^2 56.6 and 59.6, 256^2
// 82.0 and 111.9; complex64 64^2 40.3 and 10.0, 512^2 42.9 and 34.9, 768^2 71.6 and 68.3,
// 900^2 87.1 and 94.6.  (One sweep is a launch either way: 768^2 complex64 8.3 and 10.4.)
template <typename R>
int jacobi_tile_sweeps(const Op<R>& op) {
    const int limit = std::is_same<R, double>::value ? 160 : 768;
    return (op.dim == 2 && op.nbm && op.lidx && !op.face && op.n <= limit) ? kJacobiTileSweeps : 0;
}

template <typename R>
void launch_jacobi_tile(const Op<R>& op, double omega, int sweeps, const typename CT<R>::T* f,
                        const typename CT<R>::T* xin, typename CT<R>::T* xout, int conj, cudaStream_t s) {
    // about 12 x 12 blocks (one per SM), of 6 x 6 to 16 x 16 nodes (more has less halo, but a
    // node per thread)
    const int TI = std::max(6, std::min(16, (op.n + 11) / 12)), E = TI + 2 * sweeps;
    const dim3 g((op.n + TI - 1) / TI, (op.n + TI - 1) / TI), b(E, E);
    launch_after(k_jacobi_tile<R>, g, b, 2 * (size_t)E * E * sizeof(typename CT<R>::T), s, op, (R)omega, sweeps, f, xin, xout, conj);
}

template int jacobi_tile_sweeps<double>(const Op<double>&);
template int jacobi_tile_sweeps<float>(const Op<float>&);
template void launch_jacobi_tile<double>(const Op<double>&, double, int, const double2*, const double2*, double2*, int,
                                         cudaStream_t);
template void launch_jacobi_tile<float>(const Op<float>&, double, int, const float2*, const float2*, float2*, int,
                                        cudaStream_t);

template <typename R>
void launch_rbgs_half(const Op<R>& op, int colour, const typename CT<R>::T* f, typename CT<R>::T* x, int conj,
                      bool xzero, cudaStream_t s, double omega) {
    if constexpr (std::is_same<R, float>::value) {
        if (pair_ok(op, f, x, nullptr)) {
            int zc;
            const dim3 g = pair_grid(op.n, &zc), b(BX, BY);
            const float4* f4 = reinterpret_cast<const float4*>(f);
            float4* x4 = reinterpret_cast<float4*>(x);
            if (xzero) launch_after(k_rbgs_c64<true>, g, b, 0, s, op, zc, colour, f4, x4, conj, (float)omega);
            else launch_after(k_rbgs_c64<false>, g, b, 0, s, op, zc, colour, f4, x4, conj, (float)omega);
            return;
        }
    }
    const unsigned g = flat_blocks((op.N + 1) / 2);
    const bool sor = (R)omega != (R)1;
    if (xzero) launch_after(k_rbgs<R, true>, g, BX * BY, 0, s, op, colour, f, x, conj, (R)omega, sor);
    else launch_after(k_rbgs<R, false>, g, BX * BY, 0, s, op, colour, f, x, conj, (R)omega, sor);
}

bool launch_red_residual32(const Op<float>& op, const float2* f, const float2* x, float2* r_red, int conj,
                           cudaStream_t s) {
    if (!pair_ok(op, f, x, r_red)) return false;
    int zc;
    const dim3 g = pair_grid(op.n, &zc), b(BX, BY);
    launch_after(k_march_c64<2, false, false>, g, b, 0, s, op, zc, 0.f, reinterpret_cast<const float4*>(x),
                                                 reinterpret_cast<const float4*>(f), reinterpret_cast<float4*>(r_red),
                                                 nullptr, conj, Dot32{}, NormTail{});
    return true;
}

int launch_apply32_bicg(const Op<float>& op, int mode, const float2* x, float2* y, const float2* w, int conj,
                        const double2* sc, float* parts, cudaStream_t s) {
    if (!pair_ok(op, x, y, w) || (mode != 1 && mode != 2)) return 0;
    int zc;
    const dim3 g = pair_grid(op.n, &zc), b(BX, BY);
    const Dot32 d{reinterpret_cast<const float4*>(w), const_cast<double2*>(sc), parts};
    const float4* x4 = reinterpret_cast<const float4*>(x);
    float4* y4 = reinterpret_cast<float4*>(y);
    if (mode == 1) launch_after(k_march_c64<0, false, false, 1>, g, b, 0, s, op, zc, 0.f, x4, nullptr, y4, nullptr, conj, d, NormTail{});
    else launch_after(k_march_c64<0, false, false, 2>, g, b, 0, s, op, zc, 0.f, x4, nullptr, y4, nullptr, conj, d, NormTail{});
    return (int)(g.x * g.y * g.z);
}

namespace {

using SweepFn = void (*)(Op<float>, int, int, const float4*, const float2*, float2*, int, float);
template <bool K2>
SweepFn sweep_fn(bool xzero, bool sor, bool cin, bool cout) {
    if (sor) return xzero ? k_sweep_c64<true, true, K2, false, false> : k_sweep_c64<false, true, K2, false, false>;
    if (xzero) return cout ? k_sweep_c64<true, false, K2, false, true> : k_sweep_c64<true, false, K2, false, false>;
    if (cin) return cout ? k_sweep_c64<false, false, K2, true, true> : k_sweep_c64<false, false, K2, true, false>;
    return cout ? k_sweep_c64<false, false, K2, false, true> : k_sweep_c64<false, false, K2, false, false>;
}

// the nodes of one colour, one float2 per pair
__global__ void __launch_bounds__(256) k_pack_colour(int n, int colour, const float4* __restrict__ x,
                                                     float2* __restrict__ out, unsigned npairs) {
    pdl_begin();
    const unsigned h = n / 2;
    for (unsigned q = blockIdx.x * 256 + threadIdx.x; q < npairs; q += gridDim.x * 256) {
        const unsigned row = q / h, k = row / n, j = row - k * n;
        const float4 v = x[HCHK(q, npairs)];
        out[HCHK(q, npairs)] = ((j + k + colour) & 1) ? hi2(v) : lo2(v);
    }
}

}  // namespace

// Launch shape of k_sweep_c64 on an n^3 grid: whole rows per block (n/2 pairs, at most
// 128), 8, 16 or 32 rows (two of them halo) and a z chunk, by the shortest estimate of
//   waves of blocks x (planes per block + 5) x time of a step,
// where a step takes 500 clocks (its loads, barrier and shared-memory round trips) or the
// issue time of the threads resident on the SM, whichever is longer, and 5 stands for the
// two recomputed planes and the start of a block.  Small grids so get short chunks and few
// rows (64^3: 2 chunks of 30 rows left 122 of 152 SMs idle), large ones whole waves
// (256^3: 4.53 waves of 16-plane chunks cost 5).
void plan_sweep32(Op<float>& op) {
    op.sw_rows = op.sw_zc = 0;
    const int n = op.n, h = n / 2;
    if (op.dim != 3 || n % 2 != 0 || h < 1 || h > 128 || op.face || !op.ncl) return;
    const int txt = (h + 31) / 32 * 32;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 152;
    double best = 0;
    if (cudaFuncSetAttribute(k_sweep_c64<false, false, false, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024) !=
        cudaSuccess)
        return;
    for (int tyt = 8; tyt <= 32 && tyt * txt <= kSweepMaxThreads; tyt *= 2) {
        int occ = 0;
        const size_t smem = sweep_smem_bytes(txt, tyt, false);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sweep_c64<false, false, false, false, false>, txt * tyt, smem) !=
                cudaSuccess ||
            occ < 1)
            continue;
        const int gy = (n + tyt - 3) / (tyt - 2);
        for (int chunks = 1; chunks <= (n + 1) / 2; ++chunks) {
            const int zc = (n + chunks - 1) / chunks;
            const long long blocks = (long long)gy * ((n + zc - 1) / zc), slots = (long long)sms * occ;
            const long long waves = (blocks + slots - 1) / slots;
            const double resident = (double)std::min<long long>(occ, (blocks + sms - 1) / sms) * txt * tyt;
            const double cost = (double)waves * (zc + 5) * std::max(500.0, 0.8 * resident);
            if (op.sw_rows == 0 || cost < best) {
                best = cost;
                op.sw_rows = tyt;
                op.sw_zc = zc;
            }
        }
    }
}

bool rbgs_sweep32_ok(const Op<float>& op, const void* f, const void* x, const void* tmp) {
    return op.sw_rows > 0 && pair_ok(op, f, x, tmp) && x != tmp;
}

bool launch_rbgs_sweep32(const Op<float>& op, int c0, const float2* f, const float2* xin, float2* xout, int conj,
                         double omega, bool cin, bool cout, cudaStream_t s) {
    if (!rbgs_sweep32_ok(op, f, xin, xout) || (omega != 1.0 && (cin || cout)) || (cin && !xin)) return false;
    const int txt = (op.n / 2 + 31) / 32 * 32, tyt = op.sw_rows;
    const dim3 g(1, (op.n + tyt - 3) / (tyt - 2), (op.n + op.sw_zc - 1) / op.sw_zc), b(txt, tyt);
    const size_t smem = sweep_smem_bytes(txt, tyt, xin == nullptr);   // at most 78 KB
    const SweepFn fn = (op.k2 ? sweep_fn<true> : sweep_fn<false>)(xin == nullptr, omega != 1.0, cin, cout);
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024) != cudaSuccess)
        return false;
    return launch_after(fn, g, b, smem, s, op, op.sw_zc, c0, reinterpret_cast<const float4*>(f), xin, xout, conj,
                        (float)omega) == cudaSuccess;
}

void launch_pack_colour(const Op<float>& op, int colour, const float2* x, float2* out, cudaStream_t s) {
    const long long np = op.N / 2;
    launch_after(k_pack_colour, dim3((unsigned)std::min<long long>((np + 255) / 256, 8 * 152)), dim3(256), 0, s, op.n,
                 colour, reinterpret_cast<const float4*>(x), out, (unsigned)np);
}

void launch_node_pack(const Op<float>& op, uint16_t* ncl, cudaStream_t s) {
    k_node_pack<<<4 * 152, 256, 0, s>>>(op.nbm, op.lidx, ncl, op.N);
}

void launch_apply_bicg_df(const Op<double>& op, const DfTab& t, int mode, const float4* x, double2* y,
                          const double2* w, int conj, double2* sc, double* parts, unsigned* counter, cudaStream_t s) {
    const int g = bicg_grid_blocks(op.dim, op.n), b = kFusedThreads;
    if (mode == 1) launch_after(k_apply_bicg_df<1, float4>, g, b, 0, s, op, t, x, y, w, conj, sc, parts, counter);
    else launch_after(k_apply_bicg_df<2, float4>, g, b, 0, s, op, t, x, y, w, conj, sc, parts, counter);
}

void launch_apply_bicg(const Op<double>& op, int mode, const double2* x, double2* y, const double2* w, int conj,
                       double2* sc, double* parts, unsigned* counter, cudaStream_t s) {
    const int g = bicg_grid_blocks(op.dim, op.n), b = kFusedThreads;
    if (mode == 1) launch_after(k_apply_bicg<1>, g, b, 0, s, op, x, y, w, conj, sc, parts, counter);
    else launch_after(k_apply_bicg<2>, g, b, 0, s, op, x, y, w, conj, sc, parts, counter);
}

template int launch_apply<double>(const Op<double>&, const double2*, const double2*, double2*, double*, int,
                                  bool, cudaStream_t, double*, unsigned*);
template int launch_apply<float>(const Op<float>&, const float2*, const float2*, float2*, double*, int, bool,
                                 cudaStream_t, double*, unsigned*);
template void launch_jacobi<double>(const Op<double>&, double, const double2*, const double2*, double2*, int,
                                    bool, cudaStream_t);
template void launch_jacobi<float>(const Op<float>&, double, const float2*, const float2*, float2*, int, bool,
                                   cudaStream_t);
template void launch_rbgs_half<double>(const Op<double>&, int, const double2*, double2*, int, bool,
                                       cudaStream_t, double);
template void launch_rbgs_half<float>(const Op<float>&, int, const float2*, float2*, int, bool, cudaStream_t,
                                      double);

void launch_residual_red(const Op<double>& op, const double2* z, const double2* v, double2* r_red, int conj,
                         cudaStream_t s) {
    launch_after(k_residual_red, flat_blocks((op.N + 1) / 2), BX * BY, 0, s, op, z, v, r_red, conj);
}

void launch_rbgs_df_first(const Op<double>& op, const DfTab& t, const double2* f, float4* fs, float4* xs, int conj,
                          cudaStream_t s) {
    k_rbgs_df_first<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, t, f, fs, xs, conj);
}

void launch_rbgs_df(const Op<double>& op, const DfTab& t, int colour, const float4* fs, float4* xs, int conj,
                    cudaStream_t s) {
    k_rbgs_df<<<grid_for(op.dim, op.n, 2, 1), dim3(BX, BY), 0, s>>>(op, t, colour, fs, xs, conj);
}

void launch_residual_red_df(const Op<double>& op, const DfTab& t, const float4* fs, const float4* xs, float4* r_red,
                            int conj, cudaStream_t s) {
    k_residual_red_df<<<grid_for(op.dim, op.n, 2, 1), dim3(BX, BY), 0, s>>>(op, t, fs, xs, r_red, conj);
}

// blocks of the cooperative cycle: one per SM (at most), 0 if the device cannot
// launch it cooperatively
int cycle_df_blocks(long long N) {
    static int sms = -1;
    if (sms < 0) {
        int dev = 0, coop = 0, occ = 0, count = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
        if (coop) {
            int o0 = 0, o1 = 0, o2 = 0;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o0, k_cycle_df<0>, kCycleThreads, 0);
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o1, k_cycle_df<1>, kCycleThreads, 0);
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o2, k_cycle_df<2>, kCycleThreads, 0);
            occ = std::min(o0, std::min(o1, o2));
        }
        sms = (coop && occ >= 1) ? count : 0;
    }
    if (sms < 1) return 0;
    const long long need = (N + kCycleThreads - 1) / kCycleThreads;
    return (int)(need < sms ? (need < 1 ? 1 : need) : sms);
}

cudaError_t launch_cycle_df(const Op<double>& op, const DfTab& t, int pre, const double2* f, const double2* v,
                            double2* w, double2* sc, double* parts, double tol_abs, float4* fs, float4* xs,
                            float4* r_red, int n_r, int conj, unsigned* bar2, int* err, unsigned spin_limit,
                            unsigned extra_arrivals, cudaStream_t s) {
    const int nb = cycle_df_blocks(op.N);
    if (nb < 1) return cudaErrorNotSupported;
    GridBar b{bar2, bar2 + 1, err, sc, spin_limit, (unsigned)nb + extra_arrivals};
    Op<double> opv = op;
    DfTab tv = t;
    const double2* fv = f;
    const double2* vv = v;
    void* args[] = {&opv, &tv, (void*)&fv, (void*)&vv, &w, &sc, &parts, &tol_abs, &fs, &xs, &r_red, &n_r, &conj, &b};
    const void* fn = pre == 0 ? (const void*)k_cycle_df<0> : pre == 1 ? (const void*)k_cycle_df<1>
                                                                      : (const void*)k_cycle_df<2>;
    return cudaLaunchCooperativeKernel(fn, dim3(nb), dim3(kCycleThreads), args, 0, s);
}

void launch_rhs(const Op<double>& op, const double2* src, const double2* g, double2* b, cudaStream_t s) {
    k_rhs<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, src, g, b);
}

void launch_layer_k2(const Op<double>& op, double k0, double strength, const double* scale, double2* k2,
                     cudaStream_t s) {
    k_layer_k2<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, k0 * k0, strength, scale, k2);
}

void launch_invd_field(const Op<double>& op, double2* invd, cudaStream_t s) {
    k_invd_field<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, invd);
}

void launch_layer_index(const Op<double>& op, uint8_t* lidx, cudaStream_t s) {
    k_layer_index<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, lidx);
}

void launch_nbr_code(const Op<double>& op, uint8_t* code, cudaStream_t s) {
    k_nbr_code<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, code);
}

void launch_face_code(const Op<double>& op, uint8_t* face, cudaStream_t s) {
    k_face_code<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, face);
}
void launch_bvp_k2(const Op<double>& op, const double2* k2phys, double k0, int neumann_top, double2* k2eff,
                   cudaStream_t s) {
    k_bvp_k2<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, k2phys, k0, neumann_top, k2eff);
}
void launch_rhs_bvp(const Op<double>& op, const double2* src, const double2* g, int neumann_top, double2* b,
                    cudaStream_t s) {
    k_rhs_bvp<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, src, g, neumann_top, b);
}

void launch_check_ring(const Op<double>& op, int* bad, cudaStream_t s) {
    k_check_ring<<<grid_for(op.dim, op.n), dim3(BX, BY), 0, s>>>(op, bad);
}

}  // namespace helm
