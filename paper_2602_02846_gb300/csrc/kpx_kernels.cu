// kpx_kernels.cu -- the sm_103a kernels of one Kino-PAX+ iteration.
//
// Launch order per iteration (all counts are read from device memory, so
// the sequence has a fixed launch shape and can be captured in a graph):
//   begin      lambda (fixed or floor(t_e/|V_A|)), slot count, tickets,
//              region-key snapshot when the capacity rule could trigger
//   propagate  Alg. 2: one thread per (active node, sample) slot
//   mark       V_U filter: a region whose key holds a candidate id marks
//              that candidate's slot in a bitmask
//   scan       winners ranked in ascending slot order (decoupled look-back)
//   append     UpdateTree (Alg. 4): winners appended at n_nodes + rank
//              (everything but the end states); capacity rule
//   stage      the kept winners re-materialised from Philox: their end
//              states and the solution update (beside append and prune in
//              the graphs)
//   prune      PruneNodes (Alg. 3) over the pre-append tree, fused with the
//              compaction of the next V_A list (Alg. 5)
//   end        counters (in the graphs: the last block of stage and prune)
#include <cuda_runtime.h>

#include "kpx_phases.cuh"

namespace kpx {

#define KPX_DISPATCH(FN, P, ...)                                                         \
    switch ((P).dyn * 2 + (P).integ) {                                                  \
        case KPX_DI6 * 2 + KPX_EULER: return FN<KPX_DI6, KPX_EULER>(P, __VA_ARGS__);         \
        case KPX_DI6 * 2 + KPX_RK4: return FN<KPX_DI6, KPX_RK4>(P, __VA_ARGS__);             \
        case KPX_DUBINS6 * 2 + KPX_EULER: return FN<KPX_DUBINS6, KPX_EULER>(P, __VA_ARGS__); \
        case KPX_DUBINS6 * 2 + KPX_RK4: return FN<KPX_DUBINS6, KPX_RK4>(P, __VA_ARGS__);     \
        case KPX_QUAD12 * 2 + KPX_EULER: return FN<KPX_QUAD12, KPX_EULER>(P, __VA_ARGS__);   \
        case KPX_QUAD12 * 2 + KPX_RK4: return FN<KPX_QUAD12, KPX_RK4>(P, __VA_ARGS__);       \
        default: return cudaErrorInvalidValue;                                          \
    }

namespace {

// The phase kernels are launched with programmatic stream serialization
// (launch_pdl): a kernel's blocks may be set up while the one before it in the
// stream drains, and wait here, at the very top of every one of them, until it
// has completed and its writes are visible; a kernel so completes only after
// all the ones before it.  Without the launch attribute the wait is empty.
// (No early launch_dependents: the next kernels' waiting blocks then sat on
// the SMs and the dependent chain slowed down, 4.09 -> 4.29 ms among 30
// columns.)  Against plain launches and a kernel of its own for the
// iteration's end: static_di 1341 -> 1151 us, plan_di_room 646 -> 625,
// plan_dubins_open -2.6 %.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The header's words that a phase starts from, read together: one round trip
// to L2 before its first dependent load, where a test of `active` ahead of the
// other reads made it two (the loads are volatile so that they stay there).
// Words that this or a concurrent kernel writes are read but not used.
template <int Q>
__device__ __forceinline__ int4 header_quad(const kpx_device_header* H) {
    int4 v;
    asm volatile("ld.global.v4.s32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(reinterpret_cast<const int4*>(H) + Q));
    return v;
}
static_assert(offsetof(kpx_device_header, status) == 0 && offsetof(kpx_device_header, active) == 4 &&
                  offsetof(kpx_device_header, iter) == 8 && offsetof(kpx_device_header, n_nodes) == 12,
              "quad 0");
static_assert(offsetof(kpx_device_header, lambda) == 20 && offsetof(kpx_device_header, va_sel) == 24, "quad 1");
static_assert(offsetof(kpx_device_header, n_slots) == 32, "quad 2");
static_assert(offsetof(kpx_device_header, n_win) == 48 && offsetof(kpx_device_header, n_kept) == 52 &&
                  offsetof(kpx_device_header, epoch) == 60,
              "quad 3");
static_assert(offsetof(kpx_device_header, win_ticket) == 72, "quad 4");

__device__ __forceinline__ int64_t quad_int64(const int4& v) {
    return (int64_t)((uint64_t)(uint32_t)v.x | (uint64_t)(uint32_t)v.y << 32);
}

// ---------------------------------------------------------------------------
// init / reset: Alg. 1 initialisation.
// ---------------------------------------------------------------------------
template <int N>
__global__ void k_init(DevParams P, int first_time) {
    float xs[N];
#pragma unroll
    for (int d = 0; d < N; ++d) xs[d] = P.start[d];
    const int root_region = region_of<N>(P, xs);
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const uint64_t root_key = pack_key(0.0f, 0u);
    for (int64_t r = tid; r < P.R; r += stride) {
        P.region_key[r] = (r == root_region) ? root_key : KEY_INF;
        P.region_owner[r] = (r == root_region) ? 0 : -1;
    }
    for (int64_t w = tid; w < P.mask_words; w += stride) P.win_mask[w] = 0u;
    if (first_time) {
        for (int64_t t = tid; t < P.n_win_tiles; t += stride) P.win_tiles[t] = 0ull;
        for (int64_t t = tid; t < P.n_prune_tiles; t += stride) P.prune_tiles[t] = 0ull;
        for (int64_t i = tid; i < P.N; i += stride) P.clean[i] = 0u;  // epoch 0 is never current
    }
    if (tid == 0) {
        kpx_device_header* H = P.hdr;
        const int32_t epoch = first_time ? 0 : H->epoch;
        memset(H, 0, sizeof(kpx_device_header));
        H->epoch = epoch;
        H->status = KPX_OK;
        H->n_nodes = 1;
        H->count_A = 1;
        H->first_solution_iter = -1;
        H->goal_key = KEY_INF;
        if (in_goal(P, xs[0], xs[1], xs[2])) {
            H->goal_key = root_key;
            H->first_solution_iter = 0;
        }
#pragma unroll
        for (int d = 0; d < N; ++d) P.x[(int64_t)d * P.N] = xs[d];
        for (int d = 0; d < P.m; ++d) P.u[(int64_t)d * P.N] = 0.0f;
        P.K[0] = 0;
        P.parent[0] = -1;
        P.key[0] = root_key;
        P.region[0] = root_region;
        P.set[0] = SET_A;
        P.icount[0] = 0;
        P.va0[0] = 0;
    }
}

// ---------------------------------------------------------------------------
// obstacle grid (broad phase), built once per create: each cell lists its
// boxes in ascending box index.
//
// One launch: a block takes GRID_THREADS / PARTS consecutive cells.  A box
// covers a box of cells, so how many of its cells lie before the block's first
// one has a closed form, and the sum over the boxes is where the block's lists
// start: no counting pass and no scan over the cells.  The block then keeps
// the boxes that meet its rows of cells (in order, by ballots), and PARTS
// threads a cell count and copy as many parts of those.  Bound: launch latency
// and three passes over the boxes from L2.  (A warp per cell over every box, twice, and a scan
// by one block took 85 us for 1,000 boxes and 41,472 cells; this takes under 15 us.)
// PARTS is 4 while that gives every SM a block, else 32: large boxes make few
// cells with long lists (creating a planner with 1,000 boxes half as wide as the
// workspace: 177 us with 4, 101 with 32; 127 with a warp per cell as above; with
// 6,000 boxes 848, 386 and 386).
// ---------------------------------------------------------------------------
constexpr int GRID_THREADS = 256;

// the cell range of box b: lo x, y, z, hi x, y, z
__device__ __forceinline__ void box_range(const DevParams& P, int b, int (&r)[6]) {
    const float4 lo = P.obs[2 * b], hi = P.obs[2 * b + 1];
    const float l[3] = {lo.x, lo.y, lo.z}, h[3] = {hi.x, hi.y, hi.z};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        r[a] = grid_cell(l[a], P.ws_lo[a], P.grid_inv[a], P.grid_n[a]);
        r[3 + a] = grid_cell(h[a], P.ws_lo[a], P.grid_inv[a], P.grid_n[a]);
    }
}

template <int PARTS>
__global__ void __launch_bounds__(GRID_THREADS) k_grid_build(DevParams P) {
    constexpr int CELLS = GRID_THREADS / PARTS;
    constexpr int LIST = 1024;  // boxes listed at a time
    __shared__ uint32_t s_warp[GRID_THREADS / 32];
    __shared__ uint16_t s_box[LIST];
    __shared__ uint32_t s_lo[LIST], s_hi[LIST];  // their ranges, a byte an axis
    static_assert(GRID_MAX_AXIS <= 256, "a cell index fits a byte");
    const int nx = P.grid_n[0], ny = P.grid_n[1];
    const int c0 = blockIdx.x * CELLS;
    const int c1 = min(c0 + CELLS, P.n_cells) - 1;  // the block's last cell
    const int fx = c0 % nx, fy = c0 / nx % ny, fz = c0 / (nx * ny);
    const int ly = c1 / nx % ny, lz = c1 / (nx * ny);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // where the block's lists start, and (from the last block) end
    uint32_t before = 0, all = 0;
#pragma unroll 4
    for (int b = threadIdx.x; b < P.n_obs; b += GRID_THREADS) {
        int r[6];
        box_range(P, b, r);
        const int wx = r[3] - r[0] + 1, wy = r[4] - r[1] + 1;
        int n = max(min(r[5], fz - 1) - r[2] + 1, 0) * wy * wx;  // whole layers below the first cell's
        if (r[2] <= fz && fz <= r[5]) {
            n += max(min(r[4], fy - 1) - r[1] + 1, 0) * wx;      // whole rows
            if (r[1] <= fy && fy <= r[4]) n += max(min(r[3], fx - 1) - r[0] + 1, 0);
        }
        before += (uint32_t)n;
        all += (uint32_t)(wx * wy * (r[5] - r[2] + 1));
    }
    uint32_t start, total;
    block_exclusive_scan<GRID_THREADS>(before, start, s_warp);
    block_exclusive_scan<GRID_THREADS>(all, total, s_warp);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        P.cell_start[P.n_cells] = (int32_t)total;
        if ((int64_t)total > (int64_t)P.grid_cap) {
            set_status(P.hdr, KPX_E_INTERNAL);
            P.hdr->err_info[2] = total;
        }
    }
    const int c = c0 + (int)threadIdx.x / PARTS, part = (int)threadIdx.x % PARTS;
    const uint32_t cx = (uint32_t)(c % nx), cy = (uint32_t)(c / nx % ny), cz = (uint32_t)(c / (nx * ny));
    uint32_t at_cell = 0;  // pass 1: the cell's next entry
    for (int pass = 0; pass < 2; ++pass) {  // count, then copy
        uint32_t n = 0;  // pass 0: this thread's entries
        int b0 = 0;
        while (b0 < P.n_obs) {
            // the next boxes that meet the block's rows, LIST at most
            int listed = 0;
            for (; b0 < P.n_obs && listed + GRID_THREADS <= LIST; b0 += GRID_THREADS) {
                const int b = b0 + (int)threadIdx.x;
                int r[6] = {};
                bool in = false;
                if (b < P.n_obs) {
                    box_range(P, b, r);
                    in = r[2] <= lz && r[5] >= fz && (fz != lz || (r[1] <= ly && r[4] >= fy));
                }
                const uint32_t bal = __ballot_sync(FULL, in);
                if (lane == 0) s_warp[warp] = (uint32_t)__popc(bal);
                __syncthreads();
                int at = listed + __popc(bal & ((1u << lane) - 1u));
                for (int w = 0; w < GRID_THREADS / 32; ++w) {
                    if (w < warp) at += (int)s_warp[w];
                    listed += (int)s_warp[w];
                }
                if (in) {
                    s_box[at] = (uint16_t)b;
                    s_lo[at] = (uint32_t)(r[0] | r[1] << 8 | r[2] << 16);
                    s_hi[at] = (uint32_t)(r[3] | r[4] << 8 | r[5] << 16);
                }
                __syncthreads();
            }
            // this thread's part of the list
            const int l0 = listed * part / PARTS, l1 = listed * (part + 1) / PARTS;
            auto lists = [&](int l) {
                const uint32_t lo = s_lo[l], hi = s_hi[l];
                return cx >= (lo & 255u) && cx <= (hi & 255u) && cy >= (lo >> 8 & 255u) && cy <= (hi >> 8 & 255u) &&
                       cz >= lo >> 16 && cz <= hi >> 16;
            };
            uint32_t k = 0;
            for (int l = l0; l < l1; ++l) k += lists(l) ? 1u : 0u;
            n += k;
            if (pass == 1) {
                // the parts in order, behind the cell's entries of earlier lists
                uint32_t upto = k;
#pragma unroll
                for (int o = 1; o < PARTS; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(FULL, upto, o, PARTS);
                    if (part >= o) upto += y;
                }
                uint32_t at = at_cell + upto - k;
                for (int l = l0; l < l1 && c <= c1; ++l)
                    if (lists(l)) {
                        if (at < (uint32_t)P.grid_cap) {
                            const int b = s_box[l];
                            P.cell_box[2 * (int64_t)at] = P.obs[2 * b];
                            P.cell_box[2 * (int64_t)at + 1] = P.obs[2 * b + 1];
                        }
                        ++at;
                    }
                at_cell += __shfl_sync(FULL, upto, PARTS - 1, PARTS);
            }
            __syncthreads();  // the list is rewritten for the next boxes, or the next pass
        }
        if (pass == 0) {
            uint32_t sum;
            if (c > c1) n = 0;
            const uint32_t pos = start + block_exclusive_scan<GRID_THREADS>(n, sum, s_warp);
            at_cell = __shfl_sync(FULL, pos, 0, PARTS);
            const uint32_t end = __shfl_sync(FULL, pos + n, PARTS - 1, PARTS);
            if (c <= c1 && part == 0) {
                P.cell_start[c] = (int32_t)at_cell;
                P.cell_pair[c] = make_int2((int32_t)at_cell, (int32_t)min(end, (uint32_t)P.grid_cap));
            }
        }
    }
}

// ---------------------------------------------------------------------------
// begin: branching factor, slot count, tickets; region snapshot for the
// capacity rule (only when an overflow is possible this iteration).
// ---------------------------------------------------------------------------
// In the loop body of a planner's graph (loop = 1) an iteration runs only
// while iterations are owed (graph_pending > 0); otherwise every kernel of
// the iteration is a no-op.
// Every warp also sorts chunks of the iteration's slots by their order key
// (order_chunk: K, or the quadcopter's predicted step count) for the
// propagate kernel (slot_order); the slot count and lambda it uses are read
// from counters begin_counters leaves alone (|V_A|, the iteration, the V_A
// buffer), exactly as begin_counters derives them.
__global__ void k_begin(DevParams P, int loop) {
    pdl_enter();
    kpx_device_header* H = P.hdr;
    (void)header_quad<0>(H);  // with the next one: the reads below then hit L1
    (void)header_quad<1>(H);
    const bool allowed = !loop || H->graph_pending > 0;
    const bool snap = begin_needs_snapshot(P, H, allowed);  // reads counters begin_counters leaves alone
    const bool runs = allowed && problem_runs(P, H);
    const int count_A = H->count_A;
    const uint32_t iter = (uint32_t)H->iter;
    const int32_t* va = va_current(P, H);
    if (blockIdx.x == 0 && threadIdx.x == 0) begin_counters(P, H, allowed);
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (snap)
        for (int64_t r = tid; r < P.R; r += stride) P.region_snap[r] = P.region_key[r];
    if (runs && P.slot_order) {
        const int lam = begin_lambda(P, count_A);
        const int64_t n_slots = (int64_t)count_A * lam;
        const int64_t n_chunks = (n_slots + ORDER_CHUNK - 1) / ORDER_CHUNK;
        const int64_t warps = stride >> 5;
        for (int64_t c = tid >> 5; c < n_chunks; c += warps) {
            if (P.m == 4)
                order_chunk<4>(P, va, lam, iter, n_slots, c);
            else
                order_chunk<3>(P, va, lam, iter, n_slots, c);
        }
    }
}

// ---------------------------------------------------------------------------
// propagate (Alg. 2): warps take 32-slot chunks; a warp's first chunk is
// fixed (warp-major across blocks, no atomic), later chunks come from a
// ticket, so warps that drew short rollouts take more work.
// ---------------------------------------------------------------------------
template <int DYN, int INTEG, bool SYM>
__global__ void __launch_bounds__(PropShape<DYN>::threads, PropShape<DYN>::blocks)
    k_propagate(DevParams P, kpx_debug_records rec, int rec_on) {
    pdl_enter();
    kpx_device_header* H = P.hdr;
    const int4 h0 = header_quad<0>(H), h1 = header_quad<1>(H), h2 = header_quad<2>(H);
    if (!h0.y) return;  // not active
    const int64_t n_slots = quad_int64(h2);
    const int lam = h1.y;
    const uint32_t iter = (uint32_t)h0.z;
    const int32_t* va = h1.z ? P.va1 : P.va0;  // va_current()
    const bool early = (P.flags & KPX_FLAG_EARLY_REJECT) && !rec_on;
    const int64_t n_warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const bool ordered = P.slot_order != nullptr;
    const int64_t n_units = propagate_units(n_slots, ordered);  // longest first when ordered
    int64_t q = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    uint32_t steps = 0, tests = 0, n_valid = 0;
    while (q < n_units) {
        const int64_t chunk = propagate_unit_chunk(q, n_slots, ordered);
        propagate_chunk<DYN, INTEG, SYM>(P, n_slots, lam, iter, va, early, chunk, rec, rec_on, steps, tests, n_valid,
                                         P.slot_order);
        unsigned long long t = 0ull;
        if ((threadIdx.x & 31) == 0) t = atomicAdd((unsigned long long*)&H->prop_ticket, 1ull);
        q = n_warps + (int64_t)__shfl_sync(FULL, t, 0);
    }
    flush_propagate_counters(H, steps, tests, n_valid);
}

__global__ void k_mark(DevParams P) {
    pdl_enter();
    const int active = P.hdr->active;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < P.R; r += gridDim.x * blockDim.x) {
        const uint64_t k = P.region_key[r];  // with the header's word, not after it
        if (!active) return;
        mark_region(P, r, k);
    }
}

__global__ void __launch_bounds__(WIN_THREADS) k_scan(DevParams P) {
    pdl_enter();
    __shared__ uint32_t s_tile, s_prefix;
    __shared__ uint32_t s_warp[WIN_THREADS / 32];
    kpx_device_header* H = P.hdr;
    const int4 h0 = header_quad<0>(H), h2 = header_quad<2>(H), h3 = header_quad<3>(H);
    if (!h0.y) return;
    const uint32_t epoch = (uint32_t)h3.w;
    const int64_t live_words = (quad_int64(h2) + 31) / 32;
    const int per = scan_words_per_thread(P, live_words);
    const int64_t n_tiles = scan_tiles(live_words, per);
    if ((int64_t)blockIdx.x >= n_tiles) return;  // the other blocks take every tile
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(&H->win_ticket, 1u);
        __syncthreads();
        const uint32_t tile = s_tile;
        __syncthreads();
        if ((int64_t)tile >= n_tiles) return;
        scan_tile(P, H, tile, n_tiles, live_words, per, epoch, s_warp, s_prefix);
        if (n_tiles <= (int64_t)gridDim.x) return;  // a tile a block: no second ticket
    }
}

template <int DYN, int INTEG>
__global__ void __launch_bounds__(128) k_append(DevParams P) {
    pdl_enter();
    kpx_device_header* H = P.hdr;
    const int4 h0 = header_quad<0>(H), h1 = header_quad<1>(H), h3 = header_quad<3>(H);
    if (!h0.y) return;
    const int W = h3.x;
    const int n_old = h0.w;
    const int room = P.N - n_old;
    const int kept = W < room ? W : room;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        H->n_kept = kept;
        if (W > kept) set_status(H, KPX_TREE_FULL);
        // the winner scan is over: its ticket word holds prune's tile count,
        // which a prune block must not derive from the tree size (a block
        // that starts late may find the iteration already ended)
        H->win_ticket = (uint32_t)((n_old + kept + PRUNE_TILE - 1) / PRUNE_TILE);
    }
    const int lam = h1.y;
    const uint32_t iter = (uint32_t)h0.z;
    const int32_t* va = h1.z ? P.va1 : P.va0;
    for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < W; w += gridDim.x * blockDim.x)
        append_meta<DYN, INTEG>(P, H, w, kept, n_old, lam, iter, va);
}

// The end of an iteration in the loop body of a planner's graph, by the last
// working block of stage and prune to finish (no kernel of its own: 2.3 us and
// a kernel boundary per iteration).  Called by one block; `blocks`: the working
// blocks of both launches, which each caller derives from the iteration's
// winners and tiles before it reports.  The count is kept in graph_ctl, which
// is 0 between iterations.
// An iteration that ran (graph_pending > 0, as k_begin saw it) ends and is
// counted off; once the problem has stopped (tree full, an error, its
// iteration limit) the iterations still owed would be no-ops and are
// dropped.  The body's last iteration lets the loop run again while
// iterations are owed.  graph_pending only falls, so the loop ends.
__device__ __forceinline__ void finish_block(const DevParams& P, const LoopEnd& E, int blocks) {
    if (E.mode == 0) return;
    __syncthreads();
    if (threadIdx.x != 0) return;
    kpx_device_header* H = P.hdr;
    __threadfence();
    if (atomicAdd(&H->graph_ctl, 1) != blocks - 1) return;
    __threadfence();
    H->graph_ctl = 0;
    if (H->graph_pending > 0) {
        end_counters(P, H);
        H->graph_pending = problem_runs(P, H) ? H->graph_pending - 1 : 0;
    }
    if (E.mode == 2) cudaGraphSetConditional(E.handle, H->graph_pending > 0 ? 1u : 0u);
}

// The blocks of a launch that have work, at least one.
__device__ __forceinline__ int working_blocks(int grid, int64_t work) {
    return (int)(work < 1 ? 1 : (work < grid ? work : grid));
}

constexpr int STAGE_THREADS = 128;

// The kept winners' end states (one thread per winner, re-materialised) and
// the solution update; in the planner's graphs beside append and prune.
template <int DYN, int INTEG>
__global__ void __launch_bounds__(STAGE_THREADS) k_stage(DevParams P, LoopEnd E) {
    pdl_enter();
    kpx_device_header* H = P.hdr;
    const int4 h0 = header_quad<0>(H), h1 = header_quad<1>(H), h3 = header_quad<3>(H);
    if (!h0.y) {
        if (blockIdx.x == 0) finish_block(P, E, 2);
        return;
    }
    const int W = h3.x;
    const int n_old = h0.w;  // end_counters advances it only after both halves
    const int room = P.N - n_old;
    const int kept = W < room ? W : room;
    // A block that starts after the iteration's end (it has no work, so the end
    // did not wait for it) sees less room and so still no work.
    const int working = working_blocks((int)gridDim.x, (kept + STAGE_THREADS - 1) / STAGE_THREADS);
    if ((int)blockIdx.x >= working) return;
    const int lam = h1.y;
    const uint32_t iter = (uint32_t)h0.z;
    const int32_t* va = h1.z ? P.va1 : P.va0;
    const int tiles = (n_old + kept + PRUNE_TILE - 1) / PRUNE_TILE;
    for (int w = blockIdx.x * STAGE_THREADS + threadIdx.x; w < kept; w += gridDim.x * STAGE_THREADS)
        stage_winner<DYN, INTEG>(P, H, w, n_old, lam, iter, va);
    finish_block(P, E, working + working_blocks(E.prune_blocks, tiles));
}

__global__ void __launch_bounds__(PRUNE_THREADS, 8) k_prune(DevParams P, LoopEnd E) {
    pdl_enter();
    __shared__ uint32_t s_tile, s_prefix;
    __shared__ int32_t s_parent[PRUNE_TILE];
    __shared__ uint8_t s_set[PRUNE_TILE];
    __shared__ uint8_t s_icount[PRUNE_TILE];
    __shared__ uint32_t s_counts[PRUNE_ROUND_WARPS];
    kpx_device_header* H = P.hdr;
    const int4 h0 = header_quad<0>(H), h1 = header_quad<1>(H), h3 = header_quad<3>(H), h4 = header_quad<4>(H);
    if (!h0.y) {
        if (blockIdx.x == 0) finish_block(P, E, 2);
        return;
    }
    const int n_tiles = h4.z;  // append's
    if ((int)blockIdx.x >= n_tiles) return;  // the other blocks take every tile
    const int n_old = h0.w;
    const int kept = h3.y;
    const int total = n_old + kept;
    const uint32_t epoch = (uint32_t)h3.w;
    int32_t* va_next = h1.z ? P.va0 : P.va1;  // va_following()
    int cA = 0, cI = 0, cT = 0;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(&H->prune_ticket, 1u);
        __syncthreads();
        const uint32_t tile = s_tile;
        __syncthreads();
        if ((int)tile >= n_tiles) break;
        prune_tile(P, H, tile, n_tiles, n_old, total, epoch, va_next, s_parent, s_set, s_icount, s_counts, s_prefix,
                   cA, cI, cT);
        if (n_tiles <= (int)gridDim.x) break;  // a tile a block: no second ticket
    }
    flush_prune_counters(H, cA, cI, cT);
    finish_block(P, E, working_blocks((int)gridDim.x, n_tiles) +
                           working_blocks(E.stage_blocks, (kept + STAGE_THREADS - 1) / STAGE_THREADS));
}

__global__ void k_end(DevParams P) {
    pdl_enter();
    end_counters(P, P.hdr);
}

// ---------------------------------------------------------------------------
// solution extraction: parent walk from the best goal node.
// ---------------------------------------------------------------------------
__global__ void k_path(DevParams P) {
    kpx_device_header* H = P.hdr;
    const uint64_t gk = H->goal_key;
    if (gk == KEY_INF) {
        H->traj_len = -1;
        return;
    }
    const int id = (int)(uint32_t)gk;
    int len = 0;
    for (int p = id; P.parent[p] >= 0 && len < P.N; p = P.parent[p]) ++len;
    H->traj_len = len;
    int p = id;
    for (int k = len; k >= 0; --k) {
        P.path[k] = p;
        p = P.parent[p];
    }
}

__global__ void k_gather(DevParams P, int first, int rows) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    const int node = P.path[first + r];
    const int w = P.n + P.m + 1;
    float* row = P.traj + (int64_t)r * w;
    for (int d = 0; d < P.n; ++d) row[d] = P.x[(int64_t)d * P.N + node];
    for (int d = 0; d < P.m; ++d) row[P.n + d] = P.u[(int64_t)d * P.N + node];
    row[P.n + P.m] = __int_as_float((int)P.K[node]);
}

// ---------------------------------------------------------------------------
// a new region decomposition (adaptive delta): every node's region under
// the new grid; each region's key = the minimum key of its non-terminal
// nodes; a non-terminal node that does not hold its region's key is
// dominated; the memoised ancestor bits are cleared for PruneNodes to
// re-derive.  Terminal nodes keep their set byte.
// ---------------------------------------------------------------------------
__global__ void k_remap_clear(DevParams P) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < P.R; r += (int64_t)gridDim.x * blockDim.x) {
        P.region_key[r] = KEY_INF;
        P.region_owner[r] = -1;
    }
}

template <int N>
__global__ void k_remap_assign(DevParams P) {
    const int n_nodes = P.hdr->n_nodes;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_nodes; i += gridDim.x * blockDim.x) {
        float x[N];
#pragma unroll
        for (int d = 0; d < N; ++d) x[d] = P.x[(int64_t)d * P.N + i];
        const int r = region_of<N>(P, x);
        P.region[i] = r;
        if ((P.set[i] & SET_MASK) != SET_T) atomicMin((unsigned long long*)&P.region_key[r], (unsigned long long)P.key[i]);
    }
}

__global__ void k_remap_mark(DevParams P) {
    const int n_nodes = P.hdr->n_nodes;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_nodes; i += gridDim.x * blockDim.x) {
        const uint8_t sb = P.set[i];
        if ((sb & SET_MASK) == SET_T) continue;
        const int r = P.region[i];
        const bool owner = P.key[i] == P.region_key[r];
        if (owner) P.region_owner[r] = i;
        P.set[i] = (uint8_t)((sb & SET_MASK) | (owner ? 0 : SET_DOM));
    }
}

// pdl false: an ordinary launch (a kernel that joins two branches of a graph,
// or starts one)
template <typename... K, typename... A>
cudaError_t launch_kernel(bool pdl, void (*k)(K...), int grid, int block, cudaStream_t s, A... a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, K(a)...);
}

template <typename... K, typename... A>
cudaError_t launch_pdl(void (*k)(K...), int grid, int block, cudaStream_t s, A... a) {
    return launch_kernel(true, k, grid, block, s, a...);
}

int sm_count() {
    static int cached[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (!cached[dev]) {
        int sms = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cached[dev] = sms > 0 ? sms : 1;
    }
    return cached[dev];
}

// a persistent grid: enough resident blocks to fill the GPU, never more than the work
int persistent_blocks(int64_t work_blocks, int per_sm) {
    int64_t g = (int64_t)sm_count() * per_sm;
    if (g > work_blocks) g = work_blocks;
    return (int)(g < 1 ? 1 : g);
}

template <int DYN, int INTEG, bool SYM>
int propagate_blocks_per_sm() {
    static int per_sm = 0;
    if (!per_sm) {
        int v = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_propagate<DYN, INTEG, SYM>, PropShape<DYN>::threads, 0);
        per_sm = v < 1 ? 1 : v;
    }
    return per_sm;
}

template <int DYN, int INTEG>
int propagate_occupancy_t(const DevParams& P, int) {
    return P.sym_bounds ? propagate_blocks_per_sm<DYN, INTEG, true>() : propagate_blocks_per_sm<DYN, INTEG, false>();
}

int propagate_occupancy(const DevParams& P) { KPX_DISPATCH(propagate_occupancy_t, P, 0); }

template <int DYN, int INTEG>
cudaError_t launch_propagate_t(const DevParams& P, const kpx_debug_records* rec, cudaStream_t s) {
    const int fit = propagate_occupancy_t<DYN, INTEG>(P, 0);
    const int per_sm = P.prop_bps > 0 && P.prop_bps < fit ? P.prop_bps : fit;
    const int grid = persistent_blocks((P.slot_cap + PropShape<DYN>::threads - 1) / PropShape<DYN>::threads, per_sm);
    kpx_debug_records r{};
    int on = 0;
    if (rec && rec->valid) {
        r = *rec;
        on = 1;
    }
    return launch_pdl(P.sym_bounds ? k_propagate<DYN, INTEG, true> : k_propagate<DYN, INTEG, false>, grid,
                      PropShape<DYN>::threads, s, P, r, on);
}

template <int DYN, int INTEG>
cudaError_t launch_append_t(const DevParams& P, cudaStream_t s) {
    return launch_pdl(k_append<DYN, INTEG>, persistent_blocks((P.R + 127) / 128, 4), 128, s, P);
}

int stage_blocks(const DevParams& P) { return persistent_blocks((P.R + STAGE_THREADS - 1) / STAGE_THREADS, 4); }

// a tile's time is its deepest ancestor walk: as many tiles in flight as fit
// (32 registers and 6 KB of shared memory a block: 8 blocks per SM)
int prune_blocks(const DevParams& P) { return persistent_blocks(P.n_prune_tiles, 8); }

template <int DYN, int INTEG>
cudaError_t launch_stage_t(const DevParams& P, cudaStream_t s, const LoopEnd& end) {
    return launch_kernel(end.mode == 0, k_stage<DYN, INTEG>, stage_blocks(P), STAGE_THREADS, s, P, end);
}

}  // namespace

cudaError_t launch_init(const DevParams& P, bool first_time, cudaStream_t s) {
    int64_t work = P.R > P.mask_words ? P.R : P.mask_words;
    int blocks = (int)((work + 255) / 256);
    if (blocks > 2048) blocks = 2048;
    if (blocks < 1) blocks = 1;
    if (P.n == 12)
        k_init<12><<<blocks, 256, 0, s>>>(P, first_time ? 1 : 0);
    else
        k_init<6><<<blocks, 256, 0, s>>>(P, first_time ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_grid_build(const DevParams& P, cudaStream_t s) {
    if (P.n_obs == 0) return cudaSuccess;
    const auto blocks = [&](int cells) { return (P.n_cells + cells - 1) / cells; };
    if (blocks(GRID_THREADS / 4) >= sm_count())
        k_grid_build<4><<<blocks(GRID_THREADS / 4), GRID_THREADS, 0, s>>>(P);
    else
        k_grid_build<32><<<blocks(GRID_THREADS / 32), GRID_THREADS, 0, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_begin(const DevParams& P, cudaStream_t s, bool loop) {
    // the snapshot wants a few blocks per SM; the propagate order one warp
    // per 128-slot chunk (up to 6 blocks of 8 warps per SM at 40 registers)
    int64_t work = (P.R + 255) / 256;
    int per_sm = 2;
    if (P.slot_order) {
        const int64_t order_blocks = (P.slot_cap + ORDER_CHUNK * 8 - 1) / (ORDER_CHUNK * 8);
        if (order_blocks > work) work = order_blocks;
        per_sm = 6;
    }
    return launch_kernel(!loop, k_begin, persistent_blocks(work, per_sm), 256, s, P, loop ? 1 : 0);
}

cudaError_t launch_propagate(const DevParams& P, const kpx_debug_records* rec, cudaStream_t s) {
    KPX_DISPATCH(launch_propagate_t, P, rec, s);
}

cudaError_t launch_mark(const DevParams& P, cudaStream_t s) {
    return launch_pdl(k_mark, persistent_blocks((P.R + 255) / 256, 8), 256, s, P);
}

// every tile of a large iteration in flight at once (31 registers: 8 blocks per SM)
cudaError_t launch_scan(const DevParams& P, cudaStream_t s) {
    return launch_pdl(k_scan, persistent_blocks(P.n_win_tiles, 8), WIN_THREADS, s, P);
}

cudaError_t launch_append(const DevParams& P, cudaStream_t s) { KPX_DISPATCH(launch_append_t, P, s); }

LoopEnd loop_end(const DevParams& P, cudaGraphConditionalHandle h, bool last) {
    return LoopEnd{h, last ? 2 : 1, stage_blocks(P), prune_blocks(P)};
}

cudaError_t launch_stage(const DevParams& P, cudaStream_t s, const LoopEnd* end) {
    const LoopEnd e = end ? *end : LoopEnd{};
    KPX_DISPATCH(launch_stage_t, P, s, e);
}

cudaError_t launch_prune(const DevParams& P, cudaStream_t s, const LoopEnd* end) {
    return launch_pdl(k_prune, prune_blocks(P), PRUNE_THREADS, s, P, end ? *end : LoopEnd{});
}

// A look-back wait that nothing will release: tile 1 of `tiles` waits on
// tile 0 at an epoch no tile word carries.  The wait gives up after its poll
// limit and records KPX_E_TIMEOUT (err_info[0] = 0x10000 | 1): a test that the
// bounded waits end and report without faulting.
__global__ void k_wait_timeout(DevParams P, uint64_t* tiles) {
    kpx_device_header* H = P.hdr;
    uint32_t epoch = ((uint32_t)H->epoch + (1u << 29)) & 0x3FFFFFFFu;
    if (epoch == 0) epoch = 1;
    lookback(tiles, 1u, 0u, epoch, H);
}

cudaError_t launch_wait_timeout(const DevParams& P, cudaStream_t s) {
    uint64_t* tiles = P.n_win_tiles >= 2 ? P.win_tiles : (P.n_prune_tiles >= 2 ? P.prune_tiles : nullptr);
    if (!tiles) return cudaErrorInvalidValue;
    k_wait_timeout<<<1, 32, 0, s>>>(P, tiles);
    return cudaGetLastError();
}

cudaError_t launch_end(const DevParams& P, cudaStream_t s) {
    return launch_pdl(k_end, 1, 1, s, P);
}

cudaError_t launch_remap_regions(const DevParams& P, cudaStream_t s) {
    k_remap_clear<<<persistent_blocks((P.R + 255) / 256, 4), 256, 0, s>>>(P);
    const int blocks = persistent_blocks((P.N + 255) / 256, 4);
    if (P.n == 12)
        k_remap_assign<12><<<blocks, 256, 0, s>>>(P);
    else
        k_remap_assign<6><<<blocks, 256, 0, s>>>(P);
    k_remap_mark<<<blocks, 256, 0, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_path(const DevParams& P, cudaStream_t s) {
    k_path<<<1, 1, 0, s>>>(P);
    return cudaGetLastError();
}

void prepare_launches(const DevParams& P) {
    (void)sm_count();
    propagate_occupancy(P);
}

cudaError_t launch_gather(const DevParams& P, int32_t first_row, int32_t rows, cudaStream_t s) {
    if (rows <= 0) return cudaSuccess;
    k_gather<<<(rows + 127) / 128, 128, 0, s>>>(P, first_row, rows);
    return cudaGetLastError();
}

}  // namespace kpx
