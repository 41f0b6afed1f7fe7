// Compares the library's own FP64 square root and division by three with CUDA's
// correctly rounded ones on the GPU; each entry returns the number of values that differ.
#include "common.cuh"

using namespace eik;

__device__ __forceinline__ unsigned long long mix(unsigned long long x) {  // splitmix64
    x += 0x9e3779b97f4a7c15ull;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
    return x ^ (x >> 31);
}

// kind 0: random bits; 1: exponents in [-4, 4]; 2: squares of 26-bit numbers and
// their neighbours; 3: next to powers of two; 4: next to the square of a midpoint
// between two roots; 5: subnormal
__device__ double sample(unsigned long long i, int kind) {
    const unsigned long long x = mix(i);
    if (kind == 0) return __longlong_as_double((long long)(x & 0x7fffffffffffffffull));
    const long long mant = (long long)(x & 0xfffffffffffffull);
    const int e = (int)((x >> 52) % 9) - 4;
    if (kind == 1) return __longlong_as_double(((1023ll + e) << 52) | mant);
    if (kind == 5) return __longlong_as_double(mant >> (x >> 58 & 31));
    double v = 1.0;
    if (kind == 2) {
        const double s = (double)((x >> 20 & 0x3ffffff) + 1);
        v = s * s;
    } else if (kind == 3) {
        v = __longlong_as_double((1023ll + (int)(x >> 40 & 1023) - 512) << 52);
    } else {
        const double g = __longlong_as_double((1023ll << 52) | mant), u = 1.1102230246251565e-16;
        v = __fma_rn(g, g, __dmul_rn(2.0 * g, u));  // (g + ulp / 2)^2 but for the last term
    }
    return __longlong_as_double(__double_as_longlong(v) + (int)(x & 15) - 8);
}

__device__ __forceinline__ bool differ(double a, double b) {
    return __double_as_longlong(a) != __double_as_longlong(b) && !(a != a && b != b);
}

__global__ void k_root(unsigned long long n, unsigned long long seed, int kind, unsigned long long *bad) {
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const double x = sample(seed + i, kind);
        if (differ(sqrt_rn64(x), __dsqrt_rn(x))) atomicAdd(bad, 1ull);
    }
}

__global__ void k_third(unsigned long long n, unsigned long long seed, int kind, unsigned long long *bad) {
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        double x = sample(seed + i, kind);
        if (!(fabs(x) < Num<double>::inf())) continue;
        if (i & 1) x = -x;
        if (x == 0.0) x = 0.0;
        if (differ(div3(x), __ddiv_rn(x, 3.0))) atomicAdd(bad, 1ull);
    }
}

__global__ void k_third_f32(unsigned long long *bad) {  // every finite float but -0
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < (1ull << 32);
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const float x = __uint_as_float((unsigned)i);
        if (!(fabsf(x) < Num<float>::inf()) || i == 0x80000000ull) continue;
        if (__float_as_uint(div3(x)) != __float_as_uint(__fdiv_rn(x, 3.f))) atomicAdd(bad, 1ull);
    }
}

// u~ of the 2-D solve where its squares leave the range: the root of max(disc, 0)
__global__ void k_solve(unsigned long long n, unsigned long long seed, unsigned long long *bad) {
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long x = mix(seed + 3 * i);
        const double s = __longlong_as_double((long long)(1 + (x >> 20) % 2046) << 52);
        const double a = s * (1.0 + (double)(mix(x) >> 11) * 0x1p-53), b = s * (1.0 + (double)(mix(x + 1) >> 11) * 0x1p-53);
        const double rh = s * ((double)(mix(x + 2) >> 11) * 0x1p-53) * ((x & 1) ? 1.0 : 0.25);
        const double d = __dsub_rn(a, b);
        const double disc = __dsub_rn(__dmul_rn(__dmul_rn(2.0, rh), rh), __dmul_rn(d, d));
        const double u2 = __dmul_rn(__dadd_rn(__dadd_rn(a, b), __dsqrt_rn(fmax(disc, 0.0))), 0.5);
        const double want = fabs(d) < rh ? u2 : __dadd_rn(fmin(a, b), rh);
        bool two;
        if (a < Num<double>::inf() && b < Num<double>::inf() && differ(solve2(a, b, rh, two), want)) atomicAdd(bad, 1ull);
    }
}

static long long count(const void *kernel, void **args, unsigned long long **bad) {
    unsigned long long *d = nullptr, h = 0;
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return -1;
    *bad = d;
    cudaMemset(d, 0, sizeof(h));
    cudaError_t e = cudaLaunchKernel(kernel, dim3(152 * 8), dim3(256), args, 0, nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? (long long)h : -1;
}

extern "C" long long root_mismatches(unsigned long long n, unsigned long long seed, int kind) {
    unsigned long long *bad;
    void *args[] = {&n, &seed, &kind, &bad};
    return count((const void *)k_root, args, &bad);
}
extern "C" long long third_mismatches(unsigned long long n, unsigned long long seed, int kind) {
    unsigned long long *bad;
    void *args[] = {&n, &seed, &kind, &bad};
    return count((const void *)k_third, args, &bad);
}
extern "C" long long third_f32_mismatches() {
    unsigned long long *bad;
    void *args[] = {&bad};
    return count((const void *)k_third_f32, args, &bad);
}
extern "C" long long solve_mismatches(unsigned long long n, unsigned long long seed) {
    unsigned long long *bad;
    void *args[] = {&n, &seed, &bad};
    return count((const void *)k_solve, args, &bad);
}
