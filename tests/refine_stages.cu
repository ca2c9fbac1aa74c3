// One RK4 step from n states, twice: as the forward pass and the re-integration
// take it (rk4_step), and summed from the stages that the adjoint records
// (attitude_stage): by_step and by_stage[n][6], the angles and body rates.
#include "kpx_adjoint.cu"

namespace kpx {
namespace {

template <bool ISO>
__global__ void k_stage_step(RefineParams R, int n, const float* x0, const float4* u4, float* by_step,
                             float* by_stage) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float x[12], e[3], w[3];
    for (int c = 0; c < 12; ++c) x[c] = x0[12 * i + c];
    for (int a = 0; a < 3; ++a) {
        e[a] = x[3 + a];
        w[a] = x[9 + a];
    }
    const float4 v = u4[i];
    const float u[4] = {v.x, v.y, v.z, v.w};
    rk4_step<ISO>(R, x, u);
    for (int a = 0; a < 3; ++a) {
        by_step[6 * i + a] = x[3 + a];
        by_step[6 * i + 3 + a] = x[9 + a];
    }
    float es[3] = {e[0], e[1], e[2]}, ws[3] = {w[0], w[1], w[2]}, k[6], acc[6];
    for (int stage = 0; stage < 4; ++stage) {
        if (stage > 0) {
            const float hs = stage < 3 ? 0.5f * R.h : R.h;
            for (int a = 0; a < 3; ++a) {
                es[a] = fmaf(hs, k[a], e[a]);
                ws[a] = fmaf(hs, k[3 + a], w[a]);
            }
        }
        attitude_stage<ISO>(R, es, ws, v, k);
        for (int a = 0; a < 6; ++a)
            acc[a] = stage == 0 ? k[a] : (stage < 3 ? fmaf(2.0f, k[a], acc[a]) : __fadd_rn(acc[a], k[a]));
    }
    for (int a = 0; a < 6; ++a) by_stage[6 * i + a] = fmaf(R.h / 6.0f, acc[a], a < 3 ? e[a] : w[a - 3]);
}

}  // namespace
}  // namespace kpx

extern "C" int stage_steps(int n, float h, float mass, float g, const float* J, const float* x0, const float* u,
                           float* by_step, float* by_stage, void* stream) {
    kpx::RefineParams R = {};
    R.h = h;
    R.inv_mass = 1.0f / mass;
    R.g = g;
    for (int a = 0; a < 3; ++a) {
        R.J[a] = J[a];
        R.inv_J[a] = 1.0f / J[a];
    }
    const bool iso = J[0] == J[1] && J[1] == J[2];
    const auto kernel = iso ? kpx::k_stage_step<true> : kpx::k_stage_step<false>;
    kernel<<<(n + 127) / 128, 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        R, n, x0, reinterpret_cast<const float4*>(u), by_step, by_stage);
    return (int)cudaGetLastError();
}
