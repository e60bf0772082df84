// Largest deviation, in units in the last place of the IEEE result, of the
// step's fast reciprocals (lbfd_device.cuh) from 1 / x, over n arguments
// spread over the binades from 2^-emax to 2^emax.  Prints FP32 and FP64.
// Built and run by tests/test_gpu_reciprocal.py.
#include <cstdio>
#include <cstdlib>

#include "lbfd_device.cuh"

__device__ unsigned long long hash64(unsigned long long x)
{
    x ^= x >> 33;
    x *= 0xff51afd7ed558ccdull;
    x ^= x >> 33;
    x *= 0xc4ceb9fe1a85ec53ull;
    return x ^ (x >> 33);
}

__global__ void check(long long n, unsigned long long* worst)
{
    unsigned long long wf = 0, wd = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const unsigned long long h = hash64(i + 1);
        const float xf = __int_as_float((int)((h & 0x007fffffu) | ((127u - 100u + (unsigned)((h >> 32) % 201u)) << 23)));
        const int a = __float_as_int(lbfd::frcp(xf)), b = __float_as_int(1.0f / xf);
        const unsigned long long df = (unsigned long long)abs(a - b);
        wf = df > wf ? df : wf;
        const double xd = __longlong_as_double(
            (long long)((h & 0x000fffffffffffffull) | ((unsigned long long)(1023 - 900 + (int)((h >> 52) % 1801u)) << 52)));
        const long long c = __double_as_longlong(lbfd::frcp(xd)), d = __double_as_longlong(1.0 / xd);
        const unsigned long long dd = (unsigned long long)llabs(c - d);
        wd = dd > wd ? dd : wd;
    }
    atomicMax(&worst[0], wf);
    atomicMax(&worst[1], wd);
}

int main()
{
    unsigned long long *w, r[2];
    if (cudaMalloc(&w, 16) != cudaSuccess || cudaMemset(w, 0, 16) != cudaSuccess) return 1;
    check<<<304, 256>>>(1ll << 26, w);
    if (cudaMemcpy(r, w, 16, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%llu %llu\n", r[0], r[1]);
    return 0;
}
