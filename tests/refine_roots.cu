// The refinement kernels' reciprocals and roots against CUDA's correctly rounded
// ones: per check the number of values that differ and the largest difference in
// units in the last place.
#include "kpx_adjoint.cu"

namespace kpx {
namespace {

struct Tally {
    unsigned long long differ, worst;
};

__device__ void tally(Tally* t, float got, float want) {
    const int d = abs(__float_as_int(got) - __float_as_int(want));  // both positive
    if (d == 0) return;
    atomicAdd(&t->differ, 1ull);
    atomicMax(&t->worst, (unsigned long long)d);
}

__device__ uint32_t mix(uint32_t x) {
    x = (x ^ x >> 16) * 0x7FEB352Du;
    x = (x ^ x >> 15) * 0x846CA68Bu;
    return x ^ x >> 16;
}

// a value of [1, 2] by its index: its ends come up often
__device__ float one_to_two(uint32_t h) {
    const float ends[4] = {1.0f, 2.0f, __int_as_float(0x3F800001), __int_as_float(0x3FFFFFFF)};
    return h >> 28 == 0 ? ends[h & 3] : __int_as_float(0x3F800000 | (h & 0x7FFFFF));
}

__global__ void k_roots(Tally* t) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;  // < 2^24
    if (i < 1u << 23) {  // every mantissa
        const float a = __int_as_float(0x3F800000 | i);
        tally(t + 0, reciprocal(a), __frcp_rn(a));
    }
    const float b = __int_as_float(0x3F800000 + i);  // every value of [1, 4)
    tally(t + 1, root(b), __fsqrt_rn(b));
    // box_distance(): the distance and (in gx, for an offset of 1) its reciprocal
    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float gx, gy, gz;
    const float d = box_distance(2.0f, 2.0f, 2.0f, zero, zero, 1.0f, 0.0f, 0.0f, b, gx, gy, gz);
    tally(t + 2, d, __fsqrt_rn(b));
    tally(t + 3, gx, __frcp_rn(__fsqrt_rn(b)));
    // three reciprocals at once, two triples an index
    for (uint32_t k = 0; k < 2; ++k) {
        float a[3], s[3];
        for (uint32_t c = 0; c < 3; ++c) s[c] = a[c] = one_to_two(mix(i * 6u + k * 3u + c + 1u));
        reciprocals(s);
        for (uint32_t c = 0; c < 3; ++c) tally(t + 4, s[c], __frcp_rn(a[c]));
    }
}

}  // namespace
}  // namespace kpx

// out: {differ, worst} of reciprocal, root, box_distance's distance and
// reciprocal, reciprocals
extern "C" int check_roots(unsigned long long* out, void* stream) {
    kpx::k_roots<<<1 << 16, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(reinterpret_cast<kpx::Tally*>(out));
    return (int)cudaGetLastError();
}
