// SmemLimitOnce (rhd_internal.h) at a launch site of 20 kernels (the split corrector's has 18): each kernel's limit is
// raised once, whatever their number.  Prints the kernels on record after each of two rounds over all of them, and
// after the kernels' own limits are read back.  Built and run by tests/test_gpu_smem_limit.py.
#include <cstdio>
#include <utility>

#include "rhd_internal.h"

template <int I>
__global__ void kernel(float* p)
{
    extern __shared__ float s[];
    s[threadIdx.x] = (float)I;
    if (p) p[threadIdx.x] = s[threadIdx.x];
}

static rhd::SmemLimitOnce once;

template <int... I>
static bool raise_all(std::integer_sequence<int, I...>)
{
    return ((once.set(kernel<I>, 100000) == cudaSuccess) && ...);
}

template <int... I>
static int at_limit(std::integer_sequence<int, I...>)
{
    cudaFuncAttributes a;
    return ((cudaFuncGetAttributes(&a, kernel<I>) == cudaSuccess && a.maxDynamicSharedSizeBytes == 100000 ? 1 : 0) + ...);
}

int main()
{
    const auto all = std::make_integer_sequence<int, 20>{};
    if (!raise_all(all)) return 2;
    const size_t first = once.raised.size();
    if (!raise_all(all)) return 3;
    std::printf("%zu %zu %d\n", first, once.raised.size(), at_limit(all));
    return 0;
}
