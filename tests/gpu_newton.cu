// recip_newton and sqrt_newton (csrc/flbm_step.cuh) against 64-bit results and
// against CUDA's correctly rounded functions. Prints for each range the
// largest error in units of the last place against 64 bits, the largest
// distance from CUDA's result in floats, and how many differ from it.
#include <cmath>
#include <cstdio>

#include "flbm_kernels.cuh"

using namespace flbm;

struct Worst {
    unsigned long long ulp_bits;  // of a non-negative double: ordered as an integer
    unsigned long long dist, differ;
};

// Float bits first .. last in steps of stride; root: the square root.
static __global__ void sweep(unsigned first, unsigned last, unsigned stride, bool root, Worst* out)
{
    double worst = 0.0;
    unsigned long long dist = 0, differ = 0;
    const unsigned long long n = ((unsigned long long)last - first) / stride + 1;
    for (unsigned long long k = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; k < n;
         k += (unsigned long long)gridDim.x * blockDim.x) {
        const float x = __uint_as_float(first + (unsigned)(k * stride));
        const float v = root ? sqrt_newton(x) : recip_newton(x), c = root ? __fsqrt_rn(x) : __frcp_rn(x);
        const double want = root ? sqrt((double)x) : 1.0 / (double)x;
        const unsigned vb = __float_as_uint(v), cb = __float_as_uint(c);
        const unsigned long long d = vb > cb ? vb - cb : cb - vb;
        dist = d > dist ? d : dist;
        differ += d != 0;
        const double ulp = (double)__uint_as_float(cb + 1u) - (double)c;
        const double e = want == 0.0 ? fabs((double)v) : fabs((double)v - want) / ulp;
        if (!(e <= worst)) worst = e == e ? e : 1e300;
    }
    atomicMax(&out->ulp_bits, (unsigned long long)__double_as_longlong(worst));
    atomicMax(&out->dist, dist);
    atomicAdd(&out->differ, differ);
}

static bool run(const char* name, unsigned first, unsigned last, unsigned stride, bool root, Worst* dev)
{
    Worst w{};
    if (cudaMemset(dev, 0, sizeof(Worst)) != cudaSuccess) return false;
    sweep<<<1216, 256>>>(first, last, stride, root, dev);
    if (cudaMemcpy(&w, dev, sizeof(w), cudaMemcpyDeviceToHost) != cudaSuccess) return false;
    double ulp;
    std::memcpy(&ulp, &w.ulp_bits, sizeof(ulp));
    std::printf("%s ulp %.9f dist %llu differ %llu\n", name, ulp, w.dist, w.differ);
    return true;
}

int main()
{
    Worst* dev = nullptr;
    if (cudaMalloc(&dev, sizeof(Worst)) != cudaSuccess) return 2;
    bool ok = run("recip_mantissas", 0x3f800000u, 0x3fffffffu, 1u, false, dev);       // [1, 2)
    ok = ok && run("recip_range", 0x00800000u, 0x7e800000u, 509u, false, dev);        // 2^-126 .. 2^126
    ok = ok && run("root_mantissas", 0x3f800000u, 0x407fffffu, 1u, true, dev);        // [1, 4)
    ok = ok && run("root_range", 0x0d800000u, 0x7f7fffffu, 509u, true, dev);          // 2^-100 .. the largest
    ok = ok && run("root_small", 0x00000000u, 0x0d7fffffu, 1u, true, dev);            // 0 .. 2^-100
    cudaFree(dev);
    return ok ? 0 : 1;
}
