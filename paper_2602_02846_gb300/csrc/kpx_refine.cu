// kpx_refine.cu -- the C ABI of the trajectory refinement post-pass
// (include/kpx.h) and its re-validation kernel.
//
// Re-validation re-rolls each control sequence from its start state with the
// planner's own FP32 RK4 stepper.  This file has the planner's compile flags,
// so a trajectory the planner returned re-rolls to the same states bit for
// bit.  A sequence is valid when every state after a step satisfies the state
// bounds, lies in the workspace box and in no obstacle box, and the last
// position lies in the goal ball.  The edge costs are summed in FP64: FP64
// appears on the GPU only here.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "kpx_device.cuh"
#include "kpx_refine.cuh"

namespace kpx {

namespace {

struct ValidateParams {
    int32_t count, max_segments, n_obs;
    const float* obs;
    const float* x0;
    const float* u;
    const int32_t* steps;
    const int32_t* n_seg;
    int32_t* valid;
    double* cost;
    float* x_end;
};

// A block takes up to 32 trajectories.  One warp integrates them, a lane
// each, 32 steps at a time, leaving every state in shared memory; meanwhile
// sixteen warps lay out the controls of the next 32 steps and check the states
// of the previous ones (a trajectory a warp, a step a lane): bounds, then the
// boxes of the point's cell in a grid that the block builds over the workspace
// box, or every box where the grid would not pay or its lists do not fit.  The
// first state that fails ends its trajectory.  One more warp adds the FP64
// costs.  Bound: the longest trajectory's chain of RK4 steps, about 400 cycles
// each.  With a warp per trajectory, every step waiting for its 1,000 box
// tests (31 a lane), 512 sequences of up to 2,076 steps took 6.03 ms; this form
// takes 0.46 ms.  (Calls of a few steps, or among large boxes, took up to 25
// times a warp's time while every block built a grid, a warp a box and its
// size known only once it was built: 4,096 boxes over the whole workspace 2.2
// ms, now 0.05.)
constexpr int VAL_CHECK_WARPS = 16;
constexpr int VAL_COST_WARP = 4;  // on one scheduler with the integrating warp 0, which so gets the fewest checkers
constexpr int VAL_WARPS = VAL_CHECK_WARPS + 2;
constexpr int VAL_PER_WARP = 32 / VAL_CHECK_WARPS;
constexpr int VAL_ROW_BYTES = 2 * 32 * (int)(sizeof(float4) + sizeof(int) + 12 * sizeof(float));  // per trajectory
constexpr int VAL_AXIS = 16;
constexpr int VAL_CELLS = VAL_AXIS * VAL_AXIS * VAL_AXIS;
constexpr int VAL_ENTRIES = 16384;
// A block builds its grid when its trajectories have more steps than this
// together.  Both the grid and the tests it saves grow with the boxes: 4,000
// boxes of 0.02 cost it 22 us (1,000: 5 us), and testing every one of them
// costs a lone trajectory 0.4 ns a step and box, 32 trajectories of a block 0.1.
// With 4,000 boxes, grid / every box: one trajectory of 4 steps 67 / 49 us, of
// 16 72 / 78, of 32 74 / 119; four of 4 steps 71 / 53, of 16 74 / 96; 32 of 1
// step 73 / 72, of 4 73 / 114.
constexpr uint32_t VAL_GRID_STEPS = 24;
constexpr int VAL_GRID_BYTES = VAL_CELLS * (int)sizeof(int) + VAL_ENTRIES * (int)sizeof(uint16_t);

// the integrating and the checking warps, once per 32 steps
__device__ __forceinline__ void validate_barrier() {
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"((VAL_CHECK_WARPS + 1) * 32) : "memory");
}

// The block's grid over the workspace box: cell c lists boxes
// ids[c > 0 ? end[c - 1] : 0 .. end[c]), in any order.  The cell map is
// monotone, so a point in the workspace and in a box lies in a cell that
// lists the box.
struct ValGrid {
    int* end;
    uint16_t* ids;
    float inv[3];
    bool ok;  // false: the lists do not fit, every box is tested

    __device__ __forceinline__ int axis_cell(const DevParams& P, float v, int a) const {
        return grid_cell(v, P.ws_lo[a], inv[a], VAL_AXIS);
    }
};

template <bool SMEM_BOXES>
__device__ __forceinline__ void box_of(const ValidateParams& V, const float4* s_box, int b, float4& lo, float4& hi) {
    if constexpr (SMEM_BOXES) {
        lo = s_box[2 * b];
        hi = s_box[2 * b + 1];
    } else {
        const float* o = V.obs + 6 * b;
        lo = make_float4(__ldg(o), __ldg(o + 1), __ldg(o + 2), 0.0f);
        hi = make_float4(__ldg(o + 3), __ldg(o + 4), __ldg(o + 5), 0.0f);
    }
}

// The cells of box b: first cell and cells an axis (none for b past the boxes).
struct BoxCells {
    int x0, y0, z0, nx, ny, n;

    __device__ __forceinline__ int cell(int k) const {
        return ((z0 + k / (nx * ny)) * VAL_AXIS + y0 + k / nx % ny) * VAL_AXIS + x0 + k % nx;
    }
};

template <bool SMEM_BOXES>
__device__ __forceinline__ BoxCells cells_of(const DevParams& P, const ValidateParams& V, const float4* s_box,
                                             const ValGrid& G, int b) {
    BoxCells c = {};
    if (b >= V.n_obs) return c;
    float4 lo, hi;
    box_of<SMEM_BOXES>(V, s_box, b, lo, hi);
    c.x0 = G.axis_cell(P, lo.x, 0);
    c.y0 = G.axis_cell(P, lo.y, 1);
    c.z0 = G.axis_cell(P, lo.z, 2);
    c.nx = max(G.axis_cell(P, hi.x, 0) - c.x0 + 1, 0);
    c.ny = max(G.axis_cell(P, hi.y, 1) - c.y0 + 1, 0);
    c.n = c.nx * c.ny * max(G.axis_cell(P, hi.z, 2) - c.z0 + 1, 0);
    return c;
}

// Called by the whole block: a lane a box, and a box of many cells by its
// whole warp.  The cells are added up first, so lists that do not fit cost
// nothing more.
template <bool SMEM_BOXES>
__device__ void build_grid(const DevParams& P, const ValidateParams& V, const float4* s_box, ValGrid& G) {
    constexpr int THREADS = VAL_WARPS * 32, LANE_CELLS = 16;  // cells that a lane takes alone
    __shared__ int s_warp[VAL_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float w = P.ws_hi[a] - P.ws_lo[a];
        G.inv[a] = w > 0.0f ? (float)VAL_AXIS / w : 0.0f;
    }
    int total = 0;
    for (int b = threadIdx.x; b < V.n_obs; b += THREADS) total += cells_of<SMEM_BOXES>(P, V, s_box, G, b).n;
    total = __reduce_add_sync(0xFFFFFFFFu, total);
    if (lane == 0) s_warp[warp] = total;
    for (int c = threadIdx.x; c < VAL_CELLS; c += THREADS) G.end[c] = 0;
    __syncthreads();
    total = 0;
    for (int w = 0; w < VAL_WARPS; ++w) total += s_warp[w];
    G.ok = total <= VAL_ENTRIES;
    if (!G.ok) return;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {  // counts, then lists
        auto visit = [&](int b, int c) {
            const int pos = atomicAdd(&G.end[c], 1);  // second pass: from the cell's first entry on
            if (pass == 1) G.ids[pos] = (uint16_t)b;
        };
        for (int b0 = warp * 32; b0 < V.n_obs; b0 += THREADS) {
            const BoxCells m = cells_of<SMEM_BOXES>(P, V, s_box, G, b0 + lane);
            if (m.n <= LANE_CELLS)
                for (int k = 0; k < m.n; ++k) visit(b0 + lane, m.cell(k));
            for (uint32_t many = __ballot_sync(0xFFFFFFFFu, m.n > LANE_CELLS); many; many &= many - 1) {
                const int b = b0 + __ffs(many) - 1;
                const BoxCells w = cells_of<SMEM_BOXES>(P, V, s_box, G, b);
                for (int k = lane; k < w.n; k += 32) visit(b, w.cell(k));
            }
        }
        __syncthreads();
        if (pass == 1) break;
        // counts -> first entries (the second pass moves them to the ends)
        constexpr int PER = VAL_CELLS / 512;
        static_assert(THREADS >= 512, "512 threads scan the cells");
        int v[PER], sum = 0;
        const bool in = threadIdx.x < 512;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            v[q] = in ? G.end[threadIdx.x * PER + q] : 0;
            sum += v[q];
        }
        int x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        int run = x - sum;
        for (int w = 0; w < warp; ++w) run += s_warp[w];
        if (in) {
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                G.end[threadIdx.x * PER + q] = run;
                run += v[q];
            }
        }
        __syncthreads();
    }
}

// whether a point of the workspace box lies in a box that its cell lists
template <bool SMEM_BOXES>
__device__ __forceinline__ bool in_a_listed_box(const DevParams& P, const ValidateParams& V, const float4* s_box,
                                                const ValGrid& G, float px, float py, float pz) {
    const int c = (G.axis_cell(P, pz, 2) * VAL_AXIS + G.axis_cell(P, py, 1)) * VAL_AXIS + G.axis_cell(P, px, 0);
    const int e1 = G.end[c];
    bool hit = false;
    for (int e = c > 0 ? G.end[c - 1] : 0; e < e1 && !hit; ++e) {
        float4 lo, hi;
        box_of<SMEM_BOXES>(V, s_box, (int)G.ids[e], lo, hi);
        hit = px >= lo.x && px <= hi.x && py >= lo.y && py <= hi.y && pz >= lo.z && pz <= hi.z;
    }
    return hit;
}

// whether a point lies in one of the boxes first, first + stride, ...; four at
// a time, so that their loads overlap
template <bool SMEM_BOXES>
__device__ __forceinline__ bool in_a_box(const ValidateParams& V, const float4* s_box, int first, int stride, float px,
                                         float py, float pz) {
    bool hit = false;
    for (int b = first; b < V.n_obs && !hit; b += 4 * stride) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            float4 lo, hi;
            box_of<SMEM_BOXES>(V, s_box, min(b + k * stride, V.n_obs - 1), lo, hi);
            hit |= px >= lo.x && px <= hi.x && py >= lo.y && py <= hi.y && pz >= lo.z && pz <= hi.z;
        }
    }
    return hit;
}

template <bool ISO, bool SMEM_BOXES>
__global__ void __launch_bounds__(VAL_WARPS * 32, 1) k_refine_validate(DevParams P, ValidateParams V, int per_block,
                                                                      int row) {
    extern __shared__ __align__(16) unsigned char val_smem[];
    __shared__ long long s_total[32];
    __shared__ int s_done[2][32];  // 1: ended, 2: ended by a state that is not valid
    float4* su = reinterpret_cast<float4*>(val_smem);          // [chunk & 1][step][row]
    float* sx = reinterpret_cast<float*>(su + 2 * 32 * row);   // [chunk & 1][component][step][row]
    int* sseg = reinterpret_cast<int*>(sx + 2 * 12 * 32 * row);  // [chunk & 1][step][row]
    ValGrid G;
    G.end = sseg + 2 * 32 * row;
    G.ids = reinterpret_cast<uint16_t*>(G.end + VAL_CELLS);
    float4* s_box = reinterpret_cast<float4*>(val_smem + ((size_t)VAL_ROW_BYTES * row + VAL_GRID_BYTES));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * per_block;
    const int nt = (int)min((int64_t)per_block, V.count - base);
    if (SMEM_BOXES) {
        float* f = reinterpret_cast<float*>(s_box);
        for (int i = threadIdx.x; i < 6 * V.n_obs; i += VAL_WARPS * 32) {
            const int b = i / 6, c = i - 6 * b;
            f[8 * b + (c < 3 ? c : c + 1)] = V.obs[i];
        }
    }
    for (int i = warp; i < 32; i += VAL_WARPS) {
        long long t = -1;
        const int S = i < nt ? V.n_seg[base + i] : -1;
        if (S >= 0 && S <= V.max_segments) {
            t = 0;
            for (int s = lane; s < S; s += 32) t += segment_steps(V, base + i, S, s);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
        }
        if (lane == 0) {
            s_total[i] = t;  // -1: no such trajectory, or a bad segment count
            s_done[0][i] = s_done[1][i] = t > 0 ? 0 : 1;
        }
    }
    __syncthreads();
    G.ok = false;
    const uint32_t steps = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)min(max(s_total[lane], 0ll), 1ll << 20));
    if (V.n_obs > 0 && steps > VAL_GRID_STEPS) build_grid<SMEM_BOXES>(P, V, s_box, G);
    const int64_t tr = base + lane;
    if (warp == 0) {
        float x[12];
#pragma unroll
        for (int i = 0; i < 12; ++i) x[i] = lane < nt ? V.x0[tr * 12 + i] : 0.0f;
        Stepper<KPX_QUAD12, KPX_RK4> st;
        st.init(P, x, {});
        int seg = -1;
        long long left = s_total[lane];
        validate_barrier();
        for (int c = 0;; ++c) {  // chunk c; s_done[c & 1] as of the chunks before c - 1
            const bool done = s_done[c & 1][lane] != 0;
            if (__all_sync(0xFFFFFFFFu, done)) break;
            const int here = done ? 0 : (int)(left < 32 ? left : 32);
            left -= here;
            const float4* uc = su + (c & 1) * 32 * row + lane;
            const int* gs = sseg + (c & 1) * 32 * row + lane;
            float* o = sx + (c & 1) * 12 * 32 * row + lane;
            for (int t = 0; t < here; ++t) {
                const float4 v = uc[t * row];
                const float u[4] = {v.x, v.y, v.z, v.w};
                const int s = gs[t * row];
                if (s != seg) {  // a segment starts as the planner's rollouts do
                    st.init(P, x, u);
                    seg = s;
                }
                st.template advance<ISO ? 1 : 0>(P, x, u);
#pragma unroll
                for (int d = 0; d < 12; ++d) o[(d * 32 + t) * row] = x[d];
            }
            validate_barrier();
        }
        if (lane < nt && s_done[0][lane] != 2 && s_done[1][lane] != 2) {
            V.valid[tr] = s_total[lane] >= 0 && in_goal(P, x[0], x[1], x[2]) ? 1 : 0;
            if (V.x_end)
#pragma unroll
                for (int d = 0; d < 12; ++d) V.x_end[tr * 12 + d] = x[d];
        }
    } else if (warp == VAL_COST_WARP) {
        // the edge costs of every segment, in FP64 from the FP32 controls:
        // K h (1 + w e(u)); they do not depend on the states
        if (lane < nt) {
            double total = 0.0;
            const double mg = (double)P.param[0] * (double)P.param[1];
            const double tm = (double)P.param[5];
            const int S = s_total[lane] >= 0 ? V.n_seg[tr] : 0;
            for (int s = 0; s < S; ++s) {
                const float* uv = V.u + (tr * V.max_segments + s) * 4;
                const double et = ((double)uv[0] - mg) / mg;
                const double e =
                    et * et + ((double)uv[1] * uv[1] + (double)uv[2] * uv[2] + (double)uv[3] * uv[3]) / (tm * tm);
                total += (double)V.steps[tr * V.max_segments + s] * (double)P.h * (1.0 + (double)P.w_effort * e);
            }
            V.cost[tr] = total;
        }
    } else {
        const int w = warp < VAL_COST_WARP ? warp - 1 : warp - 2;
        int seg0[VAL_PER_WARP], j0[VAL_PER_WARP], done[VAL_PER_WARP], S[VAL_PER_WARP];
        long long total[VAL_PER_WARP];
#pragma unroll
        for (int k = 0; k < VAL_PER_WARP; ++k) {
            const int i = w + k * VAL_CHECK_WARPS;
            seg0[k] = j0[k] = 0;
            total[k] = s_total[i];
            done[k] = total[k] > 0 ? 0 : 1;
            S[k] = done[k] ? 0 : V.n_seg[base + i];
        }
        for (int c = -1;; ++c) {
            // c >= 0: the verdicts all warps see for chunk c (see below)
            if (c >= 0) {
                const bool all = s_done[c & 1][lane] != 0;
                if (__all_sync(0xFFFFFFFFu, all)) break;
            }
#pragma unroll
            for (int k = 0; k < VAL_PER_WARP; ++k) {
                const int i = w + k * VAL_CHECK_WARPS;
                // the controls of chunk c + 1
                const long long ahead = total[k] - 32ll * (c + 1);
                if (!done[k] && ahead > 0)
                    feed_steps(V, base + i, S[k], seg0[k], j0[k], (int)(ahead < 32 ? ahead : 32),
                               segment_steps(V, base + i, S[k], seg0[k] + lane), su + ((c + 1) & 1) * 32 * row + i,
                               sseg + ((c + 1) & 1) * 32 * row + i, row);
                // the states of chunk c - 1
                const long long back = total[k] - 32ll * (c - 1);
                if (c > 0 && !done[k]) {
                    const int n = (int)(back < 32 ? back : 32);
                    // a step a lane; without a grid the boxes of few steps
                    // are dealt out to lanes `lanes` apart
                    const int lanes = G.ok || n > 16 ? 32 : 1 << (32 - __clz(n - 1));
                    const int step = lane & (lanes - 1);
                    const float* o = sx + (((c - 1) & 1) * 12 * 32 + step) * row + i;
                    float x[12];
#pragma unroll
                    for (int d = 0; d < 12; ++d) x[d] = o[d * 32 * row];
                    bool bad = false;
                    if (step < n) {
                        bad = !bounds_ok<12>(P, x);
                        if (!bad)
                            bad = G.ok ? in_a_listed_box<SMEM_BOXES>(P, V, s_box, G, x[0], x[1], x[2])
                                       : in_a_box<SMEM_BOXES>(V, s_box, lane / lanes, 32 / lanes, x[0], x[1], x[2]);
                    }
                    for (int l = lanes; l < 32; l *= 2) bad |= __shfl_xor_sync(0xFFFFFFFFu, bad, l) != 0;
                    const uint32_t b = __ballot_sync(0xFFFFFFFFu, bad);
                    if (b) {
                        done[k] = 2;
                        if (lane == __ffs(b) - 1) {  // the first state that is not valid
                            V.valid[base + i] = 0;
                            if (V.x_end)
#pragma unroll
                                for (int d = 0; d < 12; ++d) V.x_end[(base + i) * 12 + d] = x[d];
                        }
                    } else if (back <= 32) {
                        done[k] = 1;
                    }
                }
                // read by everyone in the next round; the other buffer is
                // still being read in this one
                if (lane == 0) s_done[(c + 1) & 1][i] = done[k];
            }
            validate_barrier();
        }
    }
}

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

int n_checkpoints(int32_t max_total_steps) { return (max_total_steps + REFINE_CKPT_STEPS - 1) / REFINE_CKPT_STEPS + 1; }

bool quad_rk4(const kpx_dynamics* dyn) { return dyn && dyn->kind == KPX_QUAD12 && dyn->integ == KPX_RK4; }

bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

// workspace: the box grid first, then the checkpoints
size_t grid_region() { return align256(REFINE_GRID_BYTES); }

}  // namespace
}  // namespace kpx

using namespace kpx;

extern "C" size_t kpx_refine_workspace_size(int32_t count, int32_t max_total_steps) {
    if (count < 0 || max_total_steps < 0) return 0;
    return grid_region() +
           align256((size_t)count * n_checkpoints(max_total_steps) * REFINE_CKPT_WORDS * sizeof(float));
}

extern "C" kpx_status kpx_refine_eval(const kpx_dynamics* dyn, const kpx_refine_cost* cost, const float* obstacles,
                                      int32_t n_obstacles, int32_t count, int32_t max_segments, const float* x0,
                                      const float* u, const int32_t* steps, const int32_t* n_segments,
                                      const int32_t* order, int32_t max_total_steps, float* cost_out, float* grad_u,
                                      void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!quad_rk4(dyn) || !cost || count < 0 || max_segments < 1 || max_total_steps < 0 || n_obstacles < 0 ||
        n_obstacles > REFINE_MAX_OBS || (n_obstacles > 0 && !obstacles) || !x0 || !u || !steps || !n_segments ||
        !cost_out)
        return KPX_E_INVALID;
    if (!(cost->beta > 0.0f) || !std::isfinite(cost->beta)) return KPX_E_INVALID;
    if (!aligned16(u) || (grad_u && !aligned16(grad_u))) return KPX_E_INVALID;  // float4 rows
    if (count == 0) return KPX_OK;
    if (grad_u && (!workspace || workspace_bytes < kpx_refine_workspace_size(count, max_total_steps)))
        return KPX_E_NOMEM;
    if (workspace && reinterpret_cast<uintptr_t>(workspace) % 256 != 0) return KPX_E_INVALID;
    RefineParams R;
    memset(&R, 0, sizeof(R));
    R.h = dyn->h;
    R.inv_mass = 1.0f / dyn->param[0];
    R.g = dyn->param[1];
    for (int i = 0; i < 3; ++i) {
        R.J[i] = dyn->param[2 + i];
        R.inv_J[i] = 1.0f / dyn->param[2 + i];
    }
    R.mg = dyn->param[0] * dyn->param[1];
    R.tau_max = dyn->param[5];
    R.w_obs = cost->w_obs;
    R.beta = cost->beta;
    R.inv_beta = 1.0f / cost->beta;
    R.margin = cost->margin;
    R.w_goal = cost->w_goal;
    for (int a = 0; a < 3; ++a) R.goal[a] = cost->goal[a];
    R.w_effort = cost->w_effort;
    R.count = count;
    R.max_segments = max_segments;
    R.n_obs = n_obstacles;
    R.max_total_steps = max_total_steps;
    R.n_ckpt = n_checkpoints(max_total_steps);
    R.obs = obstacles;
    R.x0 = x0;
    R.u = u;
    R.steps = steps;
    R.n_seg = n_segments;
    R.order = order;
    R.cost = cost_out;
    R.grad = grad_u;
    // the box grid when the workspace holds it (with a gradient it always does)
    if (workspace && workspace_bytes >= grid_region()) {
        char* w = reinterpret_cast<char*>(workspace);
        R.grid = reinterpret_cast<RefineGridHeader*>(w);
        R.grid_off = reinterpret_cast<int32_t*>(w + 256);
        R.grid_cubes = R.grid_off + REFINE_GRID_CELLS + 1;
        R.grid_ids = reinterpret_cast<uint16_t*>(w + 256 + REFINE_GRID_OFF_BYTES);
    }
    R.ckpt = workspace ? reinterpret_cast<float*>(reinterpret_cast<char*>(workspace) + grid_region()) : nullptr;
    return launch_refine_eval(R, reinterpret_cast<cudaStream_t>(cuda_stream)) == cudaSuccess ? KPX_OK : KPX_E_CUDA;
}

extern "C" kpx_status kpx_refine_validate(const kpx_dynamics* dyn, const kpx_workspace* ws, const float* obstacles,
                                          int32_t n_obstacles, const kpx_goal* goal, float w_effort, int32_t count,
                                          int32_t max_segments, const float* x0, const float* u,
                                          const int32_t* steps, const int32_t* n_segments, int32_t* valid,
                                          double* cost_out, float* x_end, void* cuda_stream) {
    if (!quad_rk4(dyn) || !ws || !goal || count < 0 || max_segments < 1 || n_obstacles < 0 ||
        n_obstacles > REFINE_MAX_OBS || (n_obstacles > 0 && !obstacles) || !x0 || !u || !steps || !n_segments ||
        !valid || !cost_out)
        return KPX_E_INVALID;
    if (!aligned16(u)) return KPX_E_INVALID;
    if (count == 0) return KPX_OK;
    DevParams P;
    memset(&P, 0, sizeof(P));
    fill_dynamics(P, dyn);
    for (int a = 0; a < 3; ++a) {
        P.ws_lo[a] = ws->lo[a];
        P.ws_hi[a] = ws->hi[a];
        P.goal_c[a] = goal->center[a];
    }
    set_position_box(P);
    P.goal_r2 = goal->radius * goal->radius;
    P.cost_kind = KPX_COST_EFFORT_DURATION;
    P.w_effort = w_effort;
    ValidateParams V;
    V.count = count;
    V.max_segments = max_segments;
    V.n_obs = n_obstacles;
    V.obs = obstacles;
    V.x0 = x0;
    V.u = u;
    V.steps = steps;
    V.n_seg = n_segments;
    V.valid = valid;
    V.cost = cost_out;
    V.x_end = x_end;
    // trajectories per block: as few as one block per SM needs, at most 32; the
    // boxes in shared memory where they fit beside them
    const int sms = device_sms();
    int per_block = (count + sms - 1) / sms;
    if (per_block > 32) per_block = 32;
    const int row = per_block | 1;
    const size_t boxes = (size_t)8 * n_obstacles * sizeof(float);
    size_t smem = (size_t)VAL_ROW_BYTES * row + VAL_GRID_BYTES;
    const bool smem_boxes = smem + boxes <= REFINE_SMEM_MAX;
    if (smem_boxes) smem += boxes;
    const auto kernel = P.iso_inertia ? (smem_boxes ? k_refine_validate<true, true> : k_refine_validate<true, false>)
                                      : (smem_boxes ? k_refine_validate<false, true> : k_refine_validate<false, false>);
    static std::atomic<uint64_t> done[2][2];
    if (allow_smem((const void*)kernel, smem, done[P.iso_inertia ? 1 : 0][smem_boxes]) != cudaSuccess) return KPX_E_CUDA;
    kernel<<<(count + per_block - 1) / per_block, VAL_WARPS * 32, smem, reinterpret_cast<cudaStream_t>(cuda_stream)>>>(
        P, V, per_block, row);
    return cudaGetLastError() == cudaSuccess ? KPX_OK : KPX_E_CUDA;
}

extern "C" kpx_status kpx_refine_adam(const kpx_dynamics* dyn, int32_t count, int32_t max_segments,
                                      const int32_t* n_segments, float* u, const float* grad_u, float* m1, float* m2,
                                      int32_t t, float lr, void* cuda_stream) {
    if (!quad_rk4(dyn) || count < 0 || max_segments < 1 || !n_segments || !u || !grad_u || !m1 || !m2 || t < 1 ||
        !(lr >= 0.0f))
        return KPX_E_INVALID;
    if (count == 0) return KPX_OK;
    AdamParams A;
    A.count = count;
    A.max_segments = max_segments;
    A.n_seg = n_segments;
    A.u = u;
    A.grad = grad_u;
    A.m1 = m1;
    A.m2 = m2;
    for (int c = 0; c < 4; ++c) {
        A.lo[c] = dyn->u_lo[c];
        A.hi[c] = dyn->u_hi[c];
        if (!(A.hi[c] > A.lo[c])) return KPX_E_INVALID;
    }
    A.lr = lr;
    A.b1 = 0.9f;
    A.b2 = 0.999f;
    A.eps = 1e-8f;
    A.c1 = (float)(1.0 - std::pow(0.9, (double)t));
    A.c2 = (float)(1.0 - std::pow(0.999, (double)t));
    return launch_refine_adam(A, reinterpret_cast<cudaStream_t>(cuda_stream)) == cudaSuccess ? KPX_OK : KPX_E_CUDA;
}

extern "C" kpx_status kpx_refine_keep_best(int32_t count, int32_t max_segments, const float* u, const float* cost,
                                           float* u_best, float* cost_best, void* cuda_stream) {
    if (count < 0 || max_segments < 1 || !u || !cost || !u_best || !cost_best) return KPX_E_INVALID;
    return launch_refine_keep_best(count, max_segments, u, cost, u_best, cost_best,
                                   reinterpret_cast<cudaStream_t>(cuda_stream)) == cudaSuccess
               ? KPX_OK
               : KPX_E_CUDA;
}

extern "C" kpx_status kpx_refine_counters(const void* workspace, uint64_t counters[4], void* cuda_stream) {
    if (!workspace || !counters) return KPX_E_INVALID;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
    const RefineGridHeader* H = reinterpret_cast<const RefineGridHeader*>(workspace);
    unsigned long long t[4] = {0, 0, 0, 0};
    cudaError_t e = cudaMemcpyAsync(t, H->tests, sizeof(t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return KPX_E_CUDA;
    for (int k = 0; k < 4; ++k) counters[k] = t[k];
    return KPX_OK;
}
