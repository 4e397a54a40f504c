// Compares rcp_rn and both lanes of rcp_neg (csrc/lbm_collide.cuh) with
// __frcp_rn over every mantissa at a range of exponents; prints the number of
// values compared and of mismatches.
#include <cstdio>

#include "lbm_collide.cuh"

__global__ void k_compare(int exponent, unsigned long long *bad)
{
    const unsigned m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= 1u << 23) return;
    const float v = __uint_as_float((unsigned)(exponent + 127) << 23 | m);
    const float w = __uint_as_float((unsigned)(exponent + 127) << 23 | ((1u << 23) - 1 - m));
    const float rv = __frcp_rn(v), rw = __frcp_rn(w);
    const float2 r = gblbm::rcp_neg(make_float2(-v, -w), make_float2(1.0f, 1.0f));
    const bool ok = __float_as_uint(gblbm::rcp_rn(v)) == __float_as_uint(rv) &&
                    __float_as_uint(r.x) == __float_as_uint(rv) && __float_as_uint(r.y) == __float_as_uint(rw);
    if (!ok) atomicAdd(bad, 1ull);
}

int main()
{
    unsigned long long *bad = nullptr, out = 0, n = 0;
    cudaError_t e = cudaMalloc(&bad, sizeof(out));
    if (e == cudaSuccess) e = cudaMemset(bad, 0, sizeof(out));
    for (int exponent = -120; exponent <= 120 && e == cudaSuccess; exponent += exponent >= -8 && exponent < 8 ? 1 : 16) {
        k_compare<<<(1 << 23) / 256, 256>>>(exponent, bad);
        e = cudaGetLastError();
        n += 1ull << 23;
    }
    if (e == cudaSuccess) e = cudaMemcpy(&out, bad, sizeof(out), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
        fprintf(stderr, "%s\n", cudaGetErrorString(e));
        return 1;
    }
    printf("%llu %llu\n", n, out);
    return 0;
}
