// f64_to_pair and pair_to_f64 against the conversion instructions, value by value; prints the
// number of values and of mismatches of each, and the first mismatch.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "helm_internal.cuh"

using namespace helm;

__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b) || (isnan(a) && isnan(b)); }
__device__ bool same(double a, double b) {
    return __double_as_longlong(a) == __double_as_longlong(b) || (isnan(a) && isnan(b));
}

__global__ void k_split(const double* v, long long n, unsigned long long* bad, double* first) {
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += gridDim.x * 256LL) {
        const double x = v[i];
        const float hi = __double2float_rn(x);
        const double rest = x - (double)hi;
        const float lo = x == 0.0 ? 0.f : __double2float_rn(rest);
        const float2 p = f64_to_pair(x);
        // (a zero lo may have the value's sign)
        if (!same(p.x, hi) || !(same(p.y, lo) || (p.y == 0.f && lo == 0.f)))
            if (atomicAdd(bad, 1ull) == 0) *first = x;
    }
}

__global__ void k_join(const float2* p, long long n, unsigned long long* bad, float2* first) {
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += gridDim.x * 256LL)
        if (!same(pair_to_f64(p[i].x, p[i].y), (double)p[i].x + (double)p[i].y))
            if (atomicAdd(bad, 1ull) == 0) *first = p[i];
}

static unsigned long long rng = 88172645463325252ull;
static unsigned long long rnd() {
    rng ^= rng << 13;
    rng ^= rng >> 7;
    return rng ^= rng << 17;
}
static double from_bits(unsigned long long u) {
    double d;
    memcpy(&d, &u, 8);
    return d;
}
static float from_bits32(unsigned u) {
    float f;
    memcpy(&f, &u, 4);
    return f;
}

int main() {
    std::vector<double> v;
    // mantissas: powers of two, all ones, ties at bit 28 (even and odd above it) and their
    // neighbours, carries into the next binade, exact FP32 numbers, random ones
    std::vector<unsigned long long> m;
    for (unsigned long long top : {0ull, 1ull, 2ull, 3ull, 0x7ffffeull, 0x7fffffull, 0x400000ull, 0x2aaaaaull})
        for (unsigned long long low : {0ull, 1ull, 2ull, 0x0fffffffull, 0x10000000ull, 0x10000001ull, 0x1ffffffeull, 0x1fffffffull})
            m.push_back(top << 29 | low);
    for (int q = 0; q < 400; ++q) m.push_back(rnd() >> 12);
    for (int e = 0; e < 2048; ++e)
        for (unsigned long long f : m)
            for (unsigned long long s = 0; s < 2; ++s) v.push_back(from_bits(s << 63 | (unsigned long long)e << 52 | f));
    std::vector<float2> p;
    for (int e = 0; e < 256; ++e)
        for (unsigned f : {0u, 1u, 2u, 0x7fffffu, 0x7ffffeu, 0x400000u, 0x123456u})
            for (unsigned s = 0; s < 2; ++s) {
                const float hi = from_bits32(s << 31 | (unsigned)e << 23 | f);
                // lo: nothing, units in FP64's last place and fractions of one, half and whole
                // units of FP32's last place and beyond (pairs that are not normalised), and random
                for (int d = -60; d <= 6; ++d)
                    for (unsigned g : {0u, 1u, 0x400000u, 0x7fffffu, (unsigned)(rnd() & 0x7fffffu)})
                        for (unsigned t = 0; t < 2; ++t) {
                            const int el = e + d;
                            if (el >= 0 && el < 256) p.push_back(make_float2(hi, from_bits32(t << 31 | (unsigned)el << 23 | g)));
                        }
                for (float lo : {0.f, -0.f, from_bits32(0x7f800000u), from_bits32(0xff800000u), from_bits32(0x7fc00000u)})
                    p.push_back(make_float2(hi, lo));
            }
    double* dv;
    float2* dp;
    unsigned long long* bad;
    double* fv;
    float2* fp;
    cudaMalloc(&dv, v.size() * 8);
    cudaMalloc(&dp, p.size() * 8);
    cudaMallocManaged(&bad, 16);
    cudaMallocManaged(&fv, 8);
    cudaMallocManaged(&fp, 8);
    bad[0] = bad[1] = 0;
    *fv = 0;
    *fp = make_float2(0.f, 0.f);
    cudaMemcpy(dv, v.data(), v.size() * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(dp, p.data(), p.size() * 8, cudaMemcpyHostToDevice);
    k_split<<<608, 256>>>(dv, (long long)v.size(), bad, fv);
    k_join<<<608, 256>>>(dp, (long long)p.size(), bad + 1, fp);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    printf("%zu %llu %zu %llu first %a (%a %a)\n", v.size(), bad[0], p.size(), bad[1], *fv, fp->x, fp->y);
    return 0;
}
