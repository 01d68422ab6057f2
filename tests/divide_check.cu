// csrc/divide.cuh against the device's own division, on the device; prints one
// line per check with the number of results that differ (test_gpu_divide.py).
#include <cstdio>

#include "divide.cuh"

using namespace gsis;
typedef unsigned long long u64;

__device__ u64 mix(u64 z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ double make(u64 exponent, u64 mantissa)
{
    return __longlong_as_double((long long)(exponent << 52 | (mantissa & 0xfffffffffffffull)));
}
// mantissas: any; within 64 of 0 and of all ones
__device__ u64 mantissa(u64 r, int mode) { return mode == 0 ? r : (r & 1) ? ~(r >> 1 & 63) : r >> 1 & 63; }

__global__ void check_rcp(u64* bad)
{
    const u64 n = kRcpHi - kRcpLo + 1;
    for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x) {
        const float d = __uint_as_float(kRcpLo + (unsigned)i);
        if (__float_as_uint(rcp_newton(d)) != __float_as_uint(__frcp_rn(d))) atomicAdd(bad, 1ull);
    }
}

// mode: 0 any mantissas, 1 the divisor's next to a power of two, 2 the quotient next to 1; range: all exponents
__global__ void check_ratio(u64* bad, int per, int mode, int range)
{
    const u64 id = blockIdx.x * (u64)blockDim.x + threadIdx.x;
    for (int i = 0; i < per; ++i) {
        const u64 r = mix(id * per + i), t = mix(r ^ 0x1234567);
        const u64 ed = range ? r >> 53 : 990 + (r >> 54) % 70;
        const u64 ea = range ? (t >> 53) % 2047 : ed - (mode == 2 ? 0 : (t >> 56) % 60);
        const u64 md = mantissa(r, mode == 1), ma = mode == 2 ? (md & 0xfffffffffffffull) - (t & 63) : t;
        const double d = make(ed < 2047 ? ed : 2046, md), a = i % 97 == 0 ? 0.0 : make(ea, ma);
        if (!(a < d)) continue;
        if (__double_as_longlong(ratio(a, d)) != __double_as_longlong(a / d)) atomicAdd(bad, 1ull);
    }
}

// The same modes; 1: the mesh width's mantissa next to a power of two.  Beyond
// the exponents that div_by states, the last place may differ.
__global__ void check_div_by(u64* bad, int per, int mode, int range)
{
    const u64 id = blockIdx.x * (u64)blockDim.x + threadIdx.x;
    for (int i = 0; i < per; ++i) {
        const u64 r = mix(id * per + i), t = mix(r ^ 0x7654321);
        const u64 eh = range ? 523 + (r >> 53) % 1000 : 990 + (r >> 54) % 70, ex = range ? t >> 53 : eh - (t >> 56) % 60;
        const u64 mh = mantissa(r, mode == 1), mx = mode == 2 ? mh + (t & 127) - 64 : t;
        const double h = make(eh, mh), y = 1.0 / h;
        double x = i % 97 == 0 ? 0.0 : make(ex < 2047 ? ex : 2046, mx);
        if (t >> 20 & 1) x = -x;
        const double q = x / h, ax = fabs(x), aq = fabs(q);
        if (isinf(q)) continue;
        const bool inside = x == 0.0 || (ax >= 0x1p-960 && ax <= 0x1p960 && aq >= 0x1p-1000 && aq <= 0x1p1000);
        const long long off = __double_as_longlong(div_by(x, h, y)) - __double_as_longlong(q);
        if (off < (inside ? 0 : -1) || off > (inside ? 0 : 1)) atomicAdd(bad, 1ull);
    }
}

int main()
{
    u64* bad;
    if (cudaMallocManaged(&bad, sizeof *bad) != cudaSuccess) return 1;
    auto report = [&](const char* name) {
        const cudaError_t e = cudaDeviceSynchronize();
        if (e != cudaSuccess) {
            printf("%s: %s\n", name, cudaGetErrorString(e));
            return false;
        }
        printf("%s %llu\n", name, *bad);
        *bad = 0;
        return true;
    };
    *bad = 0;
    constexpr int B = 152 * 8, T = 256, N = 400;
    check_rcp<<<B, T>>>(bad);
    if (!report("rcp")) return 1;
    for (int mode = 0; mode < 3; ++mode)
        for (int range = 0; range < 2; ++range) {
            check_ratio<<<B, T>>>(bad, N, mode, range);
            if (!report("ratio")) return 1;
            check_div_by<<<B, T>>>(bad, N, mode, range);
            if (!report("div_by")) return 1;
        }
    return 0;
}
