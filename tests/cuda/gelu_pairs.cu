// Counts the floats z of [-z_max, z_max] at which the packed GELU (two at a time, gelu2_f) and the single one
// (gelu_f, gelu_grad_f) differ in a bit, in either half of a pair.
#include "../../paper_2312_09317_gb300/csrc/cpm_mlp_internal.h"

using namespace cpmmlp;

__global__ void compare(uint32_t n, unsigned long long *differ)
{
    unsigned long long bad = 0;
    // bit patterns 0 .. n - 1 are the floats from 0 up; their negatives sit in the pair's other half, by turns
    for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < n; k += (uint64_t)gridDim.x * blockDim.x) {
        const float p = __uint_as_float((uint32_t)k), m = -p, a = k & 1 ? m : p, b = k & 1 ? p : m;
        uint64_t grad;
        const float2 y = unpack2(gelu2_f<true>(pack2(a, b), grad)), g = unpack2(grad), only = unpack2(gelu2_f(pack2(a, b)));
        const auto same = [](float u, float v) { return __float_as_uint(u) == __float_as_uint(v); };
        bad += !same(y.x, gelu_f(a)) || !same(y.y, gelu_f(b)) || !same(only.x, y.x) || !same(only.y, y.y) ||
               !same(g.x, gelu_grad_f(a)) || !same(g.y, gelu_grad_f(b));
    }
    atomicAdd(differ, bad);
}

extern "C" int gelu_pairs(unsigned long long *compared, unsigned long long *differ)
{
    union {
        float f;
        uint32_t u;
    } most;
    most.f = kGelu2Max;
    unsigned long long *d = nullptr;
    cudaError_t e = cudaMalloc(&d, sizeof *d);
    if (e == cudaSuccess) e = cudaMemset(d, 0, sizeof *d);
    if (e == cudaSuccess) {
        compare<<<152 * 8, 256>>>(most.u + 1, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(differ, d, sizeof *d, cudaMemcpyDeviceToHost);
    cudaFree(d);
    *compared = 2ull * (most.u + 1);
    return e == cudaSuccess ? 0 : 1;
}
