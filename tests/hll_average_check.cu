// The HLL flux of the split kernels where both wave speeds are zero (fp32; subcycle_pair.cuh, subcycle_split2d.cuh): the
// average (F_L + F_R) chat / 2, the sum rounded first, for random fluxes; and states that stream along a face, for which
// alone the M1 closure's speeds are zero: their fluxes are zeros.  Prints the number of values that differ, per
// function, and of streaming states whose speeds or fluxes are not zero.  Built and run by
// tests/test_gpu_hll_average.py.
#include <cstdio>
#include <random>
#include <vector>

#include "subcycle.cuh"

__global__ void check_kernel(const float4* v, float chat, float4* out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 UL = v[4 * i], UR = v[4 * i + 1], FL = v[4 * i + 2], FR = v[4 * i + 3];
    out[3 * i] = rhd::hll_pair<false>(UL, UR, FL, FR, 0.0f, 0.0f, 0.0f, 0.0f, chat);
    out[3 * i + 1] = rhd::hll4(UL, UR, FL, FR, 0.0f, 0.0f, 0.0f, 0.0f, chat);
    out[3 * i + 2] = rhd::hll2d(UL, UR, FL, FR, 0.0f, 0.0f, 0.0f, 0.0f);  // fluxes with their factor chat
}

// states with G perpendicular to x and |G| a little above E (f is clamped to 1)
__global__ void stream_kernel(const float4* v, float chat, unsigned* off, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 r = v[4 * i];
    const float E = 1.5f + r.x, len = E * (1.00001f + 0.01f * fabsf(r.y)) * rsqrtf(r.z * r.z + r.w * r.w + 1e-30f);
    const float2 e = make_float2(E, E), z = make_float2(0.f, 0.f), gy = make_float2(len * r.z, len * r.z);
    const float2 gz = make_float2(len * r.w, len * r.w), g2 = make_float2(gy.x * gy.x + gz.x * gz.x, gy.x * gy.x + gz.x * gz.x);
    float2 a, b, l1, l3;
    rhd::closure_ab_pair<0>(e, z, gy, gz, g2, chat, 0, 0, a, b, l1, l3);
    const float4 F = rhd::flux_ab<0>(make_float4(E, 0.f, gy.x, gz.x), a.x, b.x);
    if (a.x != 0.f || l1.x != 0.f || l3.x != 0.f || F.x != 0.f || F.y != 0.f || F.z != 0.f || F.w != 0.f) atomicAdd(off, 1u);
}

int main()
{
    const int n = 1 << 16;
    const float chat = 0.3f;
    std::vector<float> v(16 * n), o(12 * n);
    std::mt19937 rng(5);
    std::uniform_real_distribution<float> d(-1.0f, 1.0f);
    for (auto& x : v) x = d(rng);
    float4 *dv, *dout;
    if (cudaMalloc(&dv, 64 * n) || cudaMalloc(&dout, 48 * n)) return 2;
    cudaMemcpy(dv, v.data(), 64 * n, cudaMemcpyHostToDevice);
    check_kernel<<<(n + 255) / 256, 256>>>(dv, chat, dout, n);
    if (cudaMemcpy(o.data(), dout, 48 * n, cudaMemcpyDeviceToHost)) return 3;
    long long off[3] = {0, 0, 0};
    for (int i = 0; i < n; ++i)
        for (int q = 0; q < 4; ++q) {
            volatile float sum = v[16 * i + 8 + q] + v[16 * i + 12 + q];
            volatile float h = 0.5f * chat;
            off[0] += o[12 * i + q] != sum * h;
            off[1] += o[12 * i + 4 + q] != sum * h;
            off[2] += o[12 * i + 8 + q] != sum * 0.5f;
        }
    unsigned *dn, streams = 0;
    if (cudaMalloc(&dn, sizeof(unsigned)) || cudaMemset(dn, 0, sizeof(unsigned))) return 4;
    stream_kernel<<<(n + 255) / 256, 256>>>(dv, chat, dn, n);
    if (cudaMemcpy(&streams, dn, sizeof(unsigned), cudaMemcpyDeviceToHost)) return 5;
    std::printf("%lld %lld %lld %u\n", off[0], off[1], off[2], streams);
    return 0;
}
