// neg_rcp2 against -__frcp_rn for every FP32 value in either half, beside a half that keeps
// the pair on its short path, leaves it (out of range on either side, zero, infinity) or is not
// a number. Prints the number of differences; the exit status is 0 if there are none.
#include <cstdio>

#include "lb_packed.cuh"

using namespace lbsc::dev;

// bit for bit, except that not-a-numbers are alike
__device__ bool differ(float a, float b)
{
    return a != a || b != b ? !(a != a && b != b) : __float_as_uint(a) != __float_as_uint(b);
}

__global__ void k_rcp(unsigned long long* bad)
{
    const float others[] = {0.7f, -3.1e-38f, 0x1p-125f, 0x1.000002p-125f, 0x1p125f, 0x1.fffffep124f, 0.f,
                            1e-42f, __int_as_float(0x7f800000), __int_as_float(0x7fc00000)};
    for (unsigned long long i = blockIdx.x * 256ull + threadIdx.x; i < 1ull << 32; i += gridDim.x * 256ull) {
        const float x = __uint_as_float((unsigned)i), want = -__frcp_rn(x);
        for (float o : others) {
            const float2 a = neg_rcp2(make_float2(x, o)), b = neg_rcp2(make_float2(o, x));
            const float wo = -__frcp_rn(o);
            if (differ(a.x, want) || differ(b.y, want) || differ(a.y, wo) || differ(b.x, wo))
                atomicAdd(bad, 1ull);
        }
    }
}

int main()
{
    unsigned long long *d = nullptr, h = 0;
    if (cudaMalloc((void**)&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess)
        return 2;
    k_rcp<<<152 * 8, 256>>>(d);
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess)
        return 2;
    cudaFree(d);
    std::printf("%llu differences\n", h);
    return h != 0;
}
