// Compares the AdamW step's Newton forms (dsm_device.cuh) with CUDA's correctly rounded operations.
//   newton_check DIVISORS GROUPS
// - div_by, div_newton: all 2^23 numerator mantissas for DIVISORS divisor mantissas (2^23: every pair);
// - sqrt_newton: 0 and every mantissa at every exponent from 2^-101 to 2^124;
// - both forms of adamw_group against adamw_elem, bit for bit, on GROUPS groups of four for each of several sets of scalars, with
//   moments from every range that the group form tells apart.
// Prints the number of differences of each; every thread writes only its own counters' atomics.
#include <cstdio>
#include <cstdlib>

#include "dsm_device.cuh"

using namespace dsm;

namespace check {

__device__ unsigned long long g_bad[4];

__device__ bool same(float a, float b) {
    return __float_as_uint(a) == __float_as_uint(b) || (isnan(a) && isnan(b));
}

__global__ void check_divisions(uint32_t divisors, uint32_t stride, uint32_t a0, uint32_t na) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= divisors) return;
    uint32_t mant = i * stride + (i * 0x9E37u) % stride;
    if (i < 64) mant = i;                                            // next to 1
    else if (divisors - i <= 64) mant = (1u << 23) - (divisors - i);  // next to 2
    const float b = __uint_as_float(0x3F800000u + mant);
    const float y = float(1.0 / double(b));
    unsigned long long bad0 = 0, bad1 = 0;
    for (uint32_t j = 0; j < na; ++j) {
        const float a = __uint_as_float(0x3F800000u + a0 + j), q = __fdiv_rn(a, b);
        bad0 += !same(div_by(a, b, y), q);
        bad1 += !same(div_newton(a, b), q);
    }
    if (bad0) atomicAdd(&g_bad[0], bad0);
    if (bad1) atomicAdd(&g_bad[1], bad1);
}

__device__ float root_or_zero(float a) { return sqrt_newton(a, __fadd_rn(a, 0x1p-126f)); }  // as adamw_rest() takes it

__global__ void check_root(int exponent) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < (1u << 23); i += gridDim.x * blockDim.x) {
        const float a = __uint_as_float((uint32_t(exponent + 127) << 23) + i), root = __fsqrt_rn(a);
        if (!same(sqrt_newton(a), root) || !same(root_or_zero(a), root)) atomicAdd(&g_bad[2], 1ull);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && !same(root_or_zero(0.f), 0.f)) atomicAdd(&g_bad[2], 1ull);
}

// A float of the given class: 0 zero, 1 usual, 2 decayed or denormal, 3 anything up to infinity, 4 an end of a range.
__device__ float pick(uint64_t h, uint32_t cls, bool negative) {
    const uint32_t mant = uint32_t(h) & 0x7FFFFFu, e = uint32_t(h >> 24) & 0xFFFFu;
    uint32_t b = 0;
    switch (cls) {
        case 0: break;
        case 1: b = ((127 - 40 + e % 45) << 23) | mant; break;
        case 2: b = e % 4 == 0 ? 1 + mant % 16 : (e % 40 << 23) | mant; break;
        case 3: b = (e % 256 << 23) | (e % 256 == 255 ? 0 : mant); break;
        default: {
            const int ends[] = {-101, -100, -99, -50, -49, 20, 27, 28, 29, 41, 42, 43};
            b = (uint32_t(127 + ends[e % 12]) << 23) + (mant % 3) - 1;
        }
    }
    return __uint_as_float(b | (negative ? 0x80000000u : 0u));
}

__global__ void check_groups(AdamScalars a, uint64_t seed, uint32_t per) {
    const uint64_t id = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    for (uint32_t k = 0; k < per; ++k) {
        const uint64_t key = sm64_finalise((seed << 48) + (id * per + k + 1) * kGoldenGamma);
        // two classes a group, so that whole groups of one class and mixed ones come up
        const uint32_t c0 = uint32_t(key) % 5, c1 = uint32_t(key >> 8) % 5, mix = uint32_t(key >> 16) & 0xFFFu;
        float x[4], m[4], v[4], g[4];
        for (int j = 0; j < 4; ++j) {
            const uint64_t h = sm64_output(key, 4 * j + 1), i = sm64_output(key, 4 * j + 2);
            m[j] = pick(h, mix >> j & 1 ? c0 : c1, h >> 63);
            v[j] = pick(i, mix >> (4 + j) & 1 ? c0 : c1, false);
            // no gradient (the moments decay), or one that sets them
            g[j] = mix >> 8 & 1 ? pick(sm64_output(key, 4 * j + 3), mix >> 9 & 3, i >> 63) : 0.f;
            x[j] = mix >> 11 & 1 ? pick(sm64_output(key, 4 * j + 4), 1 + (mix >> 10 & 1), i >> 62 & 1) : -0.f;
        }
        const float lam = key >> 40 & 1 ? 0.1f : 0.f;
        float xe[4], me[4], ve[4];
        for (int j = 0; j < 4; ++j) {
            xe[j] = x[j]; me[j] = m[j]; ve[j] = v[j];
            adamw_elem(xe[j], me[j], ve[j], g[j], a, lam);
        }
        float xc[4], mc[4], vc[4];
        for (int j = 0; j < 4; ++j) { xc[j] = x[j]; mc[j] = m[j]; vc[j] = v[j]; }
        adamw_group(x, m, v, g, a, lam);
        adamw_group<true>(xc, mc, vc, g, a, lam);
        for (int j = 0; j < 4; ++j)
            if (!same(x[j], xe[j]) || !same(m[j], me[j]) || !same(v[j], ve[j]) || !same(xc[j], xe[j]) ||
                !same(mc[j], me[j]) || !same(vc[j], ve[j]))
                atomicAdd(&g_bad[3], 1ull);
    }
}

}  // namespace check

using namespace check;

int main(int argc, char** argv) {
    const uint32_t divisors = argc > 1 ? strtoul(argv[1], nullptr, 10) : 4096;
    const uint64_t groups = argc > 2 ? strtoull(argv[2], nullptr, 10) : 1 << 24;
    const uint32_t step = 1u << 14, threads = 256;
    if (divisors == 0 || divisors > (1u << 23)) return 2;
    for (uint32_t a0 = 0; a0 < (1u << 23); a0 += step)
        check_divisions<<<(divisors + threads - 1) / threads, threads>>>(divisors, (1u << 23) / divisors, a0, step);
    for (int e = -101; e <= 124; ++e) check_root<<<1216, threads>>>(e);
    // (lr 1: x shows every bit of the quotient)
    struct Set { float b1, b2, eps; double p1, p2; };
    const Set sets[] = {
        {0.9f, 0.95f, 1e-8f, 0.9, 0.95}, {0.9f, 0.999f, 1e-8f, 0, 0.5}, {0.9f, 0.95f, 1e-8f, 0, 0}, {0.f, 0.f, 1e-6f, 0, 0},
        {0.5f, 0.5f, 1e-8f, 0, 0},       {0.9f, 0.95f, 1e-15f, 0, 0},   {0.9f, 0.95f, 1.f, 0, 0},   {0.9f, 0.95f, 1000.f, 0, 0},
        {0.9f, 0.95f, 1e-30f, 0, 0},     {0.9f, 0.95f, 1e-38f, 0, 0},   {0.9f, 0.95f, 1e-42f, 0, 0}, {0.9f, 0.95f, 1e20f, 0, 0},
        {0.9f, 0.95f, 1e6f, 0.999999, 0.9999999}};
    uint64_t seed = 0;
    for (const Set& s : sets) {
        const AdamScalars a = make_adam_scalars(s.b1, s.b2, s.eps, 1.f, s.p1, s.p2);
        const uint32_t per = 64;
        const uint64_t blocks = (groups + uint64_t(per) * threads - 1) / (uint64_t(per) * threads);
        check_groups<<<static_cast<unsigned>(blocks), threads>>>(a, ++seed, per);
    }
    const cudaError_t err = cudaDeviceSynchronize();
    if (err != cudaSuccess) {
        printf("%s\n", cudaGetErrorString(err));
        return 1;
    }
    unsigned long long bad[4];
    if (cudaMemcpyFromSymbol(bad, g_bad, sizeof bad) != cudaSuccess) return 1;
    printf("div_by %llu div_newton %llu sqrt_newton %llu adamw_group %llu\n", bad[0], bad[1], bad[2], bad[3]);
    return 0;
}
