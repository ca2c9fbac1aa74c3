// kpx_refine.cuh -- a trajectory's segments as steps, shared by the refinement
// passes (kpx_adjoint.cu) and the re-validation (kpx_refine.cu): integer work
// and copies only, so the two units' floating-point flags do not matter here.
// Params holds u (float[count][max_segments][4]), steps
// (int32[count][max_segments]) and max_segments.
#pragma once

#include <atomic>
#include <cstdint>

#include <cuda_runtime.h>

namespace kpx {

// segment s's steps (none past the trajectory's S segments)
template <class Params>
__device__ __forceinline__ int segment_steps(const Params& R, int64_t tr, int S, int s) {
    return s < S ? max(R.steps[tr * R.max_segments + s], 0) : 0;
}

// One warp, a step a lane: the controls of the trajectory's next `here` (at
// most 32) steps into u_out[step * stride], their segments into seg_out
// (either may be null).  The first step is step j0 counted from the start of
// segment s0 (j0 may lie past that segment's end: it then counts on through
// the following ones); s0 and j0 move on by 32 steps.  first: this lane's
// segment_steps(s0 + lane), which the caller may load ahead of the call.
template <class Params>
__device__ __forceinline__ void feed_steps(const Params& R, int64_t tr, int S, int& s0, int& j0, int here,
                                           int first, float4* u_out, int* seg_out, int stride) {
    const int lane = threadIdx.x & 31;
    const int64_t row = tr * R.max_segments;
    int w0 = s0, cum = -j0;  // cum: where segment w0 starts, in steps from the first
    int seg = -1;
    for (;;) {  // windows of 32 segments: one, unless segments without steps fill it
        // a segment's part from the window's start on; past 32 steps only that
        // it is longer matters, and cutting it there keeps the sums small
        int P = w0 == s0 ? first : segment_steps(R, tr, S, w0 + lane);
        P = min(lane == 0 ? P + cum : P, 64);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, P, o);
            if (lane >= o) P += y;
        }  // the window's segments up to this lane's end before step P
        int n = 0;  // the window's segments that end at or before this lane's step
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xFFFFFFFFu, P, n + o - 1) <= lane) n += o;
        if (__shfl_sync(0xFFFFFFFFu, P, n) <= lane) ++n;
        if (seg < 0 && n < 32) seg = w0 + n;
        const int m = __popc(__ballot_sync(0xFFFFFFFFu, P <= 32));
        const int before = __shfl_sync(0xFFFFFFFFu, P, m > 0 ? m - 1 : 0);
        if (m < 32 || w0 + 32 >= S) {  // step 32 lies in this window, or nothing follows it
            s0 = w0 + m;
            j0 = 32 - (m > 0 ? before : cum);
            break;
        }
        cum = before;
        w0 += 32;
    }
    if (lane < here) {
        if (u_out) u_out[lane * stride] = reinterpret_cast<const float4*>(R.u)[row + seg];
        if (seg_out) seg_out[lane * stride] = seg;
    }
}

// Dynamic shared memory that a refinement kernel may be launched with: the
// 227 KB of a block less 1 KB for the kernels' static arrays.  The limit belongs
// to the function, not to the launch, so it is set to this same value by every
// caller (one that set its own call's size could lower it under another
// thread's launch), whatever this call's (the default of 48 KB is for dynamic
// and static shared memory together), and once per device: `done` holds a bit
// for each.  (Each call setting it cost 2 us of host time.)
constexpr size_t REFINE_SMEM_MAX = 226 * 1024;

inline cudaError_t allow_smem(const void* fn, size_t bytes, std::atomic<uint64_t>& done) {
    if (bytes > REFINE_SMEM_MAX) return cudaErrorInvalidValue;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;  // 0: set at every call
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)REFINE_SMEM_MAX);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
}

inline int device_sms() {
    static std::atomic<int> known[64];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    const bool keep = dev >= 0 && dev < 64;
    if (keep) sms = known[dev].load(std::memory_order_relaxed);
    if (sms > 0) return sms;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (keep && sms > 0) known[dev].store(sms, std::memory_order_relaxed);
    return sms > 0 ? sms : 1;
}

}  // namespace kpx
