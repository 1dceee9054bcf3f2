// SwiGLU's two-wide arithmetic against CUDA's correctly rounded reciprocal and the same formula one output at a time.
#include "tik_core.cuh"

namespace {

__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b) || (a != a && b != b); }

__device__ float swiglu_scalar(float g, float u) {
    const float x = __fadd_rn(1.0f, tik::ex2_ftz(__fmul_rn(g, -tik::LOG2E_F)));
    return __fmul_rn(__fmul_rn(g, __frcp_rn(x)), u);
}

// x = the floats first .. last, in the first lane ascending, in the second descending.  count[0]: reciprocals that differ
// from __frcp_rn; count[1]: approximate reciprocals that do; count[2]: floats seen
__global__ void check_rcp(unsigned first, unsigned last, unsigned long long* count) {
    unsigned differ = 0, approx = 0, seen = 0;
    const unsigned n = last - first + 1;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float x0 = __uint_as_float(first + i), x1 = __uint_as_float(last - i);
        float r0, r1;
        tik::rcp_rn_x2(x0, x1, r0, r1);
        differ += !same(r0, __frcp_rn(x0)) + !same(r1, __frcp_rn(x1));
        approx += !same(tik::rcp_approx(x0), __frcp_rn(x0));
        ++seen;
    }
    atomicAdd(&count[0], static_cast<unsigned long long>(differ));
    atomicAdd(&count[1], static_cast<unsigned long long>(approx));
    atomicAdd(&count[2], static_cast<unsigned long long>(seen));
}

// every bf16 gate, paired with one of another size, times the given up values
__global__ void check_gates(const float* up, int n_up, unsigned long long* count) {
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 65536u) return;
    const float g0 = __uint_as_float(i << 16), g1 = __uint_as_float(((i * 40503u + 12345u) & 0xffffu) << 16);
    unsigned differ = 0;
    for (int k = 0; k < n_up; ++k) {
        const float u0 = up[k], u1 = up[n_up - 1 - k];
        float o0, o1;
        tik::swiglu_value_x2(g0, g1, u0, u1, o0, o1);
        differ += !same(o0, swiglu_scalar(g0, u0)) + !same(o1, swiglu_scalar(g1, u1));
    }
    atomicAdd(&count[0], static_cast<unsigned long long>(differ));
    atomicAdd(&count[2], 1ull);
}

}  // namespace

extern "C" int swiglu_check_rcp(unsigned first, unsigned last, unsigned long long* count) {
    check_rcp<<<148 * 8, 256>>>(first, last, count);
    return static_cast<int>(cudaDeviceSynchronize());
}
extern "C" int swiglu_check_gates(const float* up, int n_up, unsigned long long* count) {
    check_gates<<<256, 256>>>(up, n_up, count);
    return static_cast<int>(cudaDeviceSynchronize());
}
