// Deep, thin recursions (fp32 TreeRNN): one thread-block cluster per group of instances, depth by depth, without a grid
// barrier.  Tokens of different instances never meet (matching needs equal tags, and a tag belongs to one instance), so the
// cells of different instances do not depend on one another.  The cells are sorted by (group of their instance, call
// depth); the 8 blocks of a cluster split the columns of the contraction and fire the cells of their group depth by depth,
// the forward pass from the deepest depth up, the gradient pass from the first narrow depth down.
//
// What bounds such a recursion is the latency of one depth (a depth of 64 chains holds 4 or 5 cells per cluster), so
// everything that is not the chain itself is taken off it:
//   * the weights stay in registers for the whole kernel (32 per contracting thread: one column x 32 of the contracted index,
//     or two x 16), read once; operand words are read by whole warps;
//   * a result is pushed into the shared memory of all blocks of the cluster (st.async), where the cell that consumes it
//     expects its operand row (CL_SLOTS rows per depth, three depths in turn), and counted in bytes on an mbarrier there:
//     the next depth starts when its rows are complete, whatever else -- stores to global memory among it -- is in flight;
//   * a helper warp fetches ahead, straight to shared memory, what does not depend on the chain: list ends, records, operand
//     rows of leaves, and for the gradient the state and dlog of the callees;
//   * a block tells the others when it has read the rows of a depth (an mbarrier in each of them), which is waited for
//     before a push two depths later: nobody runs further ahead.
// Cells of a depth beyond the first CL_SLOTS go through global memory (a cluster barrier orders those depths).
// Measured per depth, 64 chains, H = 256 (weights in shared memory and states through L2 -> this): forward 4.7 -> 1.86 us,
// gradient 5.0 -> 1.96 us.
#pragma once
#include "rdf_tc.cuh"

static const int CL_SLOTS = 16;                // cells of a depth whose operand rows live in shared memory; cells per step
static const int CL_WARPS = 16;                // contracting and finishing warps; one more fetches ahead (96 registers per thread)
static const int CL_THREADS = (CL_WARPS + 1) * 32;
static const int CL_MAX_H = 256;
static const uint32_t CL_NO_SLOT = 63u;
static const int CL_RING = 16;                 // depths whose records are in shared memory

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float sum2(f32x2 v) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    return lo + hi;
}
__device__ __forceinline__ uint32_t cl_mapa(uint32_t addr, int rank) {       // the same place in block `rank` of the cluster
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// 16 bytes into another block's shared memory, counted on the mbarrier there
__device__ __forceinline__ void cl_push(uint32_t addr, float a, float b, float c, float d, uint32_t mbar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d), "r"(mbar) : "memory");
}
__device__ __forceinline__ void cl_copy16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// a row of global memory (this GPU's) to shared memory; addresses and size are multiples of 16 bytes (H and CPC are multiples of 4)
__device__ __forceinline__ void cl_bulk(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}
// one arrival on the mbarrier of every block of the cluster that has columns (a warp: lane = block)
__device__ __forceinline__ void cl_arrive_all(uint32_t mbar, int active, int lane) {
    if (lane < active) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cl_mapa(mbar, lane)) : "memory");
}

// The warp's 32 results (lane = column; v and the lane's slot_bytes valid where `want`) to the rows of the next depth in
// every active block.  Four columns per store; to: address of (slot 0, the warp's first column) of the buffer in this block.
// Columns of one 16-byte piece share `want` and `slot_bytes`.
template <int LANES>
__device__ __forceinline__ void cl_push_row(float v, bool want, uint32_t slot_bytes, uint32_t to, uint32_t mbar, int active, int lane) {
    constexpr int PIECES = LANES / 4, RANKS = 32 / PIECES;             // lane = (piece, block); CLUSTER_CTAS / RANKS rounds
    const int src = (lane % PIECES) * 4;
    const float a = __shfl_sync(0xffffffffu, v, src), b = __shfl_sync(0xffffffffu, v, src + 1);
    const float c = __shfl_sync(0xffffffffu, v, src + 2), d = __shfl_sync(0xffffffffu, v, src + 3);
    const bool go = __shfl_sync(0xffffffffu, (int)want, src) != 0;
    const uint32_t off = __shfl_sync(0xffffffffu, slot_bytes, src) + 16u * (lane % PIECES);
#pragma unroll
    for (int r0 = 0; r0 < CLUSTER_CTAS; r0 += RANKS) {
        const int r = r0 + lane / PIECES;
        if (go && r < active) cl_push(cl_mapa(to + off, r), a, b, c, d, cl_mapa(mbar, r));
    }
}

// The contraction of N operand rows (x: the thread's slice of the first) with the block's CPC columns, partial over the
// warps: part[cell][col] = sum over the warp's k of w[col][k] x[cell][k].  thread = (column lane, and lane + 32 when there are
// 64; KPT consecutive k): the lanes of a warp read the same operand words, pairs of consecutive k share a packed
// multiply-add, and a sum needs no shuffle (one for 16 columns, whose warps hold two slices of k).
template <int CPC, int KPT, int N>
__device__ __forceinline__ void cl_mac(const f32x2 (&w)[(CPC + 31) / 32][KPT / 2], const float* x, int stride, float* part, int lane) {
    constexpr int COLS = (CPC + 31) / 32;
    f32x2 acc[N][COLS];
#pragma unroll
    for (int q = 0; q < N; ++q)
#pragma unroll
        for (int e = 0; e < COLS; ++e) acc[q][e] = 0ull;
#pragma unroll
    for (int i = 0; i < KPT / 4; ++i) {
        ulonglong2 v[N];
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] = *reinterpret_cast<const ulonglong2*>(x + (size_t)q * stride + 4 * i);
#pragma unroll
        for (int q = 0; q < N; ++q)
#pragma unroll
            for (int e = 0; e < COLS; ++e) acc[q][e] = fma2(w[e][2 * i], v[q].x, acc[q][e]);
#pragma unroll
        for (int q = 0; q < N; ++q)
#pragma unroll
            for (int e = 0; e < COLS; ++e) acc[q][e] = fma2(w[e][2 * i + 1], v[q].y, acc[q][e]);
    }
#pragma unroll
    for (int q = 0; q < N; ++q)
#pragma unroll
        for (int e = 0; e < COLS; ++e) {
            float t = sum2(acc[q][e]);
            if (CPC < 32) t += __shfl_xor_sync(0xffffffffu, t, 16);
            if (lane < CPC) part[q * CPC + 32 * e + lane] = t;
        }
}
template <int CPC, int KPT>
__device__ __forceinline__ void cl_contract(const f32x2 (&w)[(CPC + 31) / 32][KPT / 2], const float* rows, int stride, int n, float* part, int lane) {
    for (int q = 0; q < n; q += 6) {
        const float* x = rows + (size_t)q * stride;
        float* p = part + q * CPC;
        switch (min(n - q, 6)) {
            case 1: cl_mac<CPC, KPT, 1>(w, x, stride, p, lane); break;
            case 2: cl_mac<CPC, KPT, 2>(w, x, stride, p, lane); break;
            case 3: cl_mac<CPC, KPT, 3>(w, x, stride, p, lane); break;
            case 4: cl_mac<CPC, KPT, 4>(w, x, stride, p, lane); break;
            case 5: cl_mac<CPC, KPT, 5>(w, x, stride, p, lane); break;
            default: cl_mac<CPC, KPT, 6>(w, x, stride, p, lane); break;
        }
    }
}
template <int CPC>
__device__ __forceinline__ float cl_total(const float* part, int cell, int col) {       // the warps' partial sums, in order
    float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < CL_WARPS; ++w) t[w & 3] += part[((size_t)w * CL_SLOTS + cell) * CPC + col];
    return (t[0] + t[1]) + (t[2] + t[3]);
}
__device__ __forceinline__ void cl_bar_contract() { asm volatile("bar.sync 1, 512;" ::: "memory"); }     // all warps but the helper
static_assert(CL_WARPS * 32 == 512, "bar.sync 1");

// The depths of a group in the order the kernel runs them: step t.  {first cell in the sorted list, cells}
struct ClDepth {
    uint32_t begin, n;
};
struct ClRings {
    ClDepth  depth[CL_RING];
    uint4    rec[CL_RING][CL_SLOTS];           // {cell, left, right, -}
    uint4    link[CL_RING][CL_SLOTS];          // see rdf_group_kernel
    uint32_t end[CL_RING];                     // list end between steps t - 1 and t
    uint64_t rows_full[3];                     // rows of step t complete: mbarrier t % 3
    uint64_t rows_read[4];                     // rows of step t read by every block: mbarrier t % 4
};

// the last depth at which the group has cells
__device__ __forceinline__ uint32_t cl_last_depth(const uint32_t* ends, uint32_t top) {
    uint32_t lo = 0, hi = top;
    const uint32_t all = ends[top];
    while (lo < hi) {
        const uint32_t mid = (lo + hi) / 2;
        if (ends[mid] >= all) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// The helper warp's view of the steps.  Everything it fetches goes straight to shared memory (cp.async): list ends CL_ENDS
// steps ahead, records CL_RECORDS ahead, one group of copies per step, so that no load is waited for in the step that issues it.
static const int CL_ENDS = 10, CL_RECORDS = 6;
template <bool DOWN>                           // DOWN: step t is depth first + t, else depth first - t
struct ClAhead {
    const uint32_t* ends;
    uint32_t first, steps, cap;
    // list end between steps t - 1 and t
    __device__ __forceinline__ const uint32_t* end_at(uint32_t t) const { return ends + (DOWN ? first - 1u + t : first - t); }
    __device__ __forceinline__ void fetch_end(ClRings& R, uint32_t t, int lane) const {
        if (lane == 0 && t <= steps)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(&R.end[t % CL_RING])), "l"(end_at(t)) : "memory");
    }
    __device__ __forceinline__ void fetch_records(const DevCtx& c, ClRings& R, uint32_t t, int lane) const {
        ClDepth dp{0u, 0u};
        if (t < steps) {
            const uint32_t a = min(R.end[t % CL_RING], cap), b = min(R.end[(t + 1u) % CL_RING], cap);
            dp = DOWN ? ClDepth{a, b - a} : ClDepth{b, a - b};
        }
        if (lane == 0) R.depth[t % CL_RING] = dp;
        if (lane < CL_SLOTS && (uint32_t)lane < dp.n) {
            cl_copy16(smem_u32(&R.rec[t % CL_RING][lane]), &c.cell_sorted[dp.begin + lane]);
            cl_copy16(smem_u32(&R.link[t % CL_RING][lane]), &c.cell_link[dp.begin + lane]);
        }
    }
    __device__ __forceinline__ void start(const DevCtx& c, ClRings& R, int lane) const {       // records of steps 0 .. CL_RECORDS - 1
        for (uint32_t t = 0; t < (uint32_t)CL_ENDS; ++t) fetch_end(R, t, lane);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        for (uint32_t t = 0; t < (uint32_t)CL_RECORDS; ++t) fetch_records(c, R, t, lane);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
    }
    // in step t, after the rows of step t + 2 have been asked for
    __device__ __forceinline__ void advance(const DevCtx& c, ClRings& R, uint32_t t, int lane) const {
        fetch_end(R, t + CL_ENDS, lane);
        fetch_records(c, R, t + CL_RECORDS, lane);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 2;" ::: "memory");               // the groups up to step t - 2 have landed: the ends of
        __syncwarp();                                                      // step t + 7 and the records of step t + 4 among them
    }
};

// the weights of one contracting thread: at(col, k) for its columns and KPT consecutive k
template <int CPC, int KPT, class F>
__device__ __forceinline__ void cl_weights(f32x2 (&w)[(CPC + 31) / 32][KPT / 2], int warp, int lane, int k0, F at) {
#pragma unroll
    for (int e = 0; e < (CPC + 31) / 32; ++e)
#pragma unroll
        for (int i = 0; i < KPT / 2; ++i) {
            const int col = 32 * e + (CPC < 32 ? lane % CPC : lane), k = k0 + 2 * i;
            w[e][i] = warp < CL_WARPS ? pack2(at(col, k), at(col, k + 1)) : 0ull;
        }
}

// CPC columns of W per block (8 x CPC >= H), KPT contracted indices per thread (16 warps, two slices each for 16 columns: at least 2H)
template <int CPC, int KPT>
__global__ void __launch_bounds__(CL_THREADS, 1) rdf_operator_cluster_kernel(const __grid_constant__ DevCtx c) {
    constexpr int ROW = CL_WARPS * (CPC < 32 ? 2 : 1) * KPT;                        // floats per operand row (padded with zeros)
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    __shared__ ClRings R;
    // every block of the grid takes the same decision from the same words: no block of a cluster is left waiting
    if (c.ctl->forward_status != 0 || c.ctl->status != 0 || depth_groups(c) <= 1u) return;
    float* xs = reinterpret_cast<float*>(dyn_smem);                        // [3][CL_SLOTS][ROW]
    float* part = xs + (size_t)3 * CL_SLOTS * ROW;                         // [2][CL_WARPS][CL_SLOTS][CPC]
    const int H = c.H, K2 = 2 * c.H, rank = blockIdx.x % CLUSTER_CTAS, group = blockIdx.x / CLUSTER_CTAS, j0 = rank * CPC;
    const int active = (H + CPC - 1) / CPC;                                // blocks that have columns
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t top = depth_stride(c) - 1u;
    const uint32_t* ends = c.group_ends + (size_t)group * depth_stride(c);
    const uint32_t d0 = min(c.ctl->d_split, top), last = max(d0, cl_last_depth(ends, top)), steps = last - d0;   // depths last .. d0 + 1
    for (int q = threadIdx.x; q < 3 * CL_SLOTS * ROW; q += CL_THREADS) xs[q] = 0.f;
    f32x2 w[(CPC + 31) / 32][KPT / 2];
    const int k0 = (CPC < 32 ? warp * 2 + lane / 16 : warp) * KPT;
    cl_weights<CPC, KPT>(w, warp, lane, k0, [&](int col, int k) { return j0 + col < H && k < K2 ? __ldg(&c.W[(size_t)(j0 + col) * K2 + k]) : 0.f; });
    const int fcol = j0 + lane;                                            // finishing: a warp takes a cell, lane = column
    const bool fin_col = lane < CPC && fcol < H;
    const float bias = fin_col ? __ldg(&c.b[fcol]) : 0.f;
    const uint32_t full0 = smem_u32(R.rows_full), read0 = smem_u32(R.rows_read);
    if (threadIdx.x == 0) {
        for (int k = 0; k < 3; ++k) mbar_init(full0 + 8 * k, 1);           // the helper's count of bytes
        for (int k = 0; k < 4; ++k) mbar_init(read0 + 8 * k, (uint32_t)active);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");           // the zeroed rows before the bulk copies
    __syncthreads();
    // helper: the operand rows of step t (its records are in the ring), lane = (slot, port): a leaf's row is one bulk copy, a
    // cell's comes with the pushes of the step before
    auto arm = [&](uint32_t t) {
        const uint32_t n = min(R.depth[t % CL_RING].n, (uint32_t)CL_SLOTS), mbar = full0 + 8 * (t % 3u);
        const uint32_t s = lane >> 1, port = lane & 1;
        if (lane == 0) mbar_arrive_expect_tx(mbar, n * 8u * H);
        __syncwarp();
        if (s < n) {
            const uint4 rec = R.rec[t % CL_RING][s], link = R.link[t % CL_RING][s];
            if ((port ? link.y : link.x) >> 31)
                cl_bulk(smem_u32(xs + ((size_t)(t % 3u) * CL_SLOTS + s) * ROW + port * H), c.arena + (size_t)min(port ? rec.z : rec.y, c.frame_cap - 1u) * H,
                        4u * H, mbar);
        }
        __syncwarp();
    };
    const ClAhead<false> ahead{ends, last, steps, c.work_cap};
    if (warp == CL_WARPS && rank < active) {                               // (a block without columns must leave no copy in flight)
        ahead.start(c, R, lane);
        arm(0);
        arm(1);
    }
    __syncthreads();
    cluster_sync_all();                                                    // every block is set up: pushes may come
    if (rank >= active) return;                                            // (no columns; nobody pushes to it or waits for it)
    for (uint32_t t = 0; t < steps; ++t) {
        if (warp == CL_WARPS) {
            if (t) mbar_wait(c, read0 + 8 * ((t - 1u) & 3u), ((t - 1u) >> 2) & 1u);          // the rows of step t - 1 have been read (here too)
            arm(t + 2u);
            ahead.advance(c, R, t, lane);
        } else {
            mbar_wait(c, full0 + 8 * (t % 3u), (t / 3u) & 1u);
            const ClDepth dp = R.depth[t % CL_RING];
            if (dp.n == 0 && warp == 0) cl_arrive_all(read0 + 8 * (t & 3u), active, lane);   // (no cell of this group at this depth)
            float* rows = xs + (size_t)(t % 3u) * CL_SLOTS * ROW;
            float* sums = part + (size_t)(t & 1u) * CL_WARPS * CL_SLOTS * CPC;
            for (uint32_t first = 0; first < dp.n; first += CL_SLOTS) {
                const int n = (int)min((uint32_t)CL_SLOTS, dp.n - first);
                if (first) {
                    // beyond the slots: operand rows from global memory
                    cl_bar_contract();                                     // (the rows and sums of the round before are no longer read)
                    for (int s = warp; s < n; s += CL_WARPS) {
                        const uint4 rec = __ldcg(reinterpret_cast<const uint4*>(&c.cell_sorted[dp.begin + first + s]));
                        for (int p = lane; p < K2 / 4; p += 32) {
                            const int k = 4 * p;
                            const uint32_t src = k < H ? rec.y : rec.z;
                            if (src < c.frame_cap)
                                *reinterpret_cast<float4*>(rows + (size_t)s * ROW + k) = ldcg4(c.arena + (size_t)src * H + (k < H ? k : k - H));
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    cl_bar_contract();
                }
                uint32_t out = 0xFFFFFFFFu, to = 0u;                       // the cell this warp finishes, where its state goes
                if (warp < n) {
                    out = first ? __ldcg(&c.cell_sorted[dp.begin + first + warp].out) : R.rec[t % CL_RING][warp].x;
                    to = first ? __ldcg(&c.cell_link[dp.begin + first + warp].z) : R.link[t % CL_RING][warp].z;
                }
                cl_contract<CPC, KPT>(w, rows + k0, ROW, n, sums + (size_t)warp * CL_SLOTS * CPC, lane);
                cl_bar_contract();
                if (first + CL_SLOTS >= dp.n && warp == CL_WARPS - 1) cl_arrive_all(read0 + 8 * (t & 3u), active, lane);   // the rows have been read
                if (warp < n) {
                    const bool live = fin_col && out < c.frame_cap;
                    const float h = tanhf((fin_col ? cl_total<CPC>(sums, warp, lane) : 0.f) + bias);
                    if (t > 1 && first == 0) mbar_wait(c, read0 + 8 * ((t - 2u) & 3u), ((t - 2u) >> 2) & 1u);   // nobody reads step t - 2's rows any more
                    // the operand row of the cell that takes this state, in every block of the cluster
                    const uint32_t slot = to & 63u, port = (to >> 6) & 1u;
                    cl_push_row<CPC>(h, live && slot < (uint32_t)CL_SLOTS && t + 1u < steps, 4u * (slot * ROW + port * H),
                                     smem_u32(xs + (size_t)((t + 1u) % 3u) * CL_SLOTS * ROW + j0), full0 + 8 * ((t + 1u) % 3u), active, lane);
                    if (live) c.arena[(size_t)out * H + fcol] = h;
                }
            }
            __syncwarp();
        }
        if (t + 1u < steps && R.depth[(t + 1u) % CL_RING].n > (uint32_t)CL_SLOTS) {   // (the next step reads states from global memory)
            cluster_sync_all();
        }
    }
    cluster_sync_all();                                                    // (no block leaves while another may still signal it)
}

// The gradient counterpart: [dh_l ; dh_r] = W^T dz for the cells of a depth, CPC of the 2H columns per block; the thread that
// adds the sums up finishes the callee of its column (adds W_s^T dlog; a cell callee gets dz = dh (1 - h^2) as its row, a
// leaf callee adds dh to dE[tok]).
template <int CPC, int KPT>
__global__ void __launch_bounds__(CL_THREADS, 1) rdf_backward_cluster_kernel(const __grid_constant__ DevCtx c) {
    constexpr int ROW = CL_WARPS * (CPC < 32 ? 2 : 1) * KPT, CLASSES = 8, FC = (CPC + 31) / 32;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    __shared__ ClRings R;
    if (c.ctl->forward_status != 0 || c.ctl->status != 0 || depth_groups(c) <= 1u) return;
    float* zs = reinterpret_cast<float*>(dyn_smem);                        // [3][CL_SLOTS][ROW]: dz rows
    float* part = zs + (size_t)3 * CL_SLOTS * ROW;                         // [2][CL_WARPS][CL_SLOTS][CPC]
    float* hs = part + (size_t)2 * CL_WARPS * CL_SLOTS * CPC;                // [4][CL_SLOTS][CPC]: state of the callee under each column
    float* dls = hs + (size_t)4 * CL_SLOTS * CPC;                          // [4][CL_SLOTS][2][8]: dlog of both callees
    float* ws = dls + (size_t)4 * CL_SLOTS * 16;                           // [CLASSES][CPC]: W_s under the block's columns
    const int H = c.H, K2 = 2 * c.H, rank = blockIdx.x % CLUSTER_CTAS, group = blockIdx.x / CLUSTER_CTAS, j0 = rank * CPC;
    const int active = (K2 + CPC - 1) / CPC;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t top = depth_stride(c) - 1u;
    const uint32_t* ends = c.group_ends + (size_t)group * depth_stride(c);
    const uint32_t d0 = min(c.ctl->d_split, top), last = max(d0, cl_last_depth(ends, top)), steps = last - d0;   // depths d0 + 1 .. last
    for (int q = threadIdx.x; q < 3 * CL_SLOTS * ROW; q += CL_THREADS) zs[q] = 0.f;
    for (int q = threadIdx.x; q < CLASSES * CPC; q += CL_THREADS) {
        const int k = q / CPC, col = j0 + q % CPC;
        ws[q] = col < K2 && k < c.n_classes ? __ldg(&c.W_s[k * H + (col < H ? col : col - H)]) : 0.f;
    }
    f32x2 w[(CPC + 31) / 32][KPT / 2];
    const int k0 = (CPC < 32 ? warp * 2 + lane / 16 : warp) * KPT;
    cl_weights<CPC, KPT>(w, warp, lane, k0, [&](int col, int k) { return j0 + col < K2 && k < H ? __ldg(&c.W[(size_t)k * K2 + j0 + col]) : 0.f; });
    const uint32_t full0 = smem_u32(R.rows_full), read0 = smem_u32(R.rows_read);
    if (threadIdx.x == 0) {
        for (int k = 0; k < 3; ++k) mbar_init(full0 + 8 * k, 1);
        for (int k = 0; k < 4; ++k) mbar_init(read0 + 8 * k, (uint32_t)active);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");           // the zeroed rows before the bulk copies
    __syncthreads();
    // helper: what the finishing threads of step t need of the callees, lane = (slot, callee); the dz rows themselves come
    // from the step before (the first ones from global memory, where the grid-wide kernel left them)
    const int c_lo = (lane & 1) ? max(j0, H) : j0, c_hi = min((lane & 1) ? K2 : H, j0 + CPC);      // columns of this block that belong to the lane's callee
    auto arm = [&](uint32_t t) {
        const uint32_t n = min(R.depth[t % CL_RING].n, (uint32_t)CL_SLOTS), mbar = full0 + 8 * (t % 3u);
        const uint32_t s = lane >> 1, which = lane & 1, ring = (t % 4u) * CL_SLOTS + s;
        if (lane == 0) mbar_arrive_expect_tx(mbar, n * (64u + 4u * (min(K2, j0 + CPC) - j0) + 4u * H));
        __syncwarp();
        if (s < n) {
            const uint4 rec = R.rec[t % CL_RING][s];
            const uint32_t ch = min(which ? rec.z : rec.y, c.frame_cap - 1u);
            cl_bulk(smem_u32(dls + (size_t)(ring * 2 + which) * 8), c.dlog + (size_t)ch * 8, 32u, mbar);
            if (c_hi > c_lo) cl_bulk(smem_u32(hs + (size_t)ring * CPC + (c_lo - j0)), c.arena + (size_t)ch * H + (c_lo - (which ? H : 0)), 4u * (c_hi - c_lo), mbar);
            if (t == 0 && which == 0) cl_bulk(smem_u32(zs + (size_t)s * ROW), c.dhp + (size_t)min(rec.x, c.frame_cap - 1u) * H, 4u * H, mbar);
        }
        __syncwarp();
    };
    const ClAhead<true> ahead{ends, d0 + 1u, steps, c.work_cap};
    if (warp == CL_WARPS && rank < active) {                               // (a block without columns must leave no copy in flight)
        ahead.start(c, R, lane);
        arm(0);
        arm(1);
    }
    __syncthreads();
    cluster_sync_all();
    if (rank >= active) return;
    for (uint32_t t = 0; t < steps; ++t) {
        if (warp == CL_WARPS) {
            if (t) mbar_wait(c, read0 + 8 * ((t - 1u) & 3u), ((t - 1u) >> 2) & 1u);
            arm(t + 2u);
            ahead.advance(c, R, t, lane);
        } else {
            mbar_wait(c, full0 + 8 * (t % 3u), (t / 3u) & 1u);
            const ClDepth dp = R.depth[t % CL_RING];
            if (dp.n == 0 && warp == 0) cl_arrive_all(read0 + 8 * (t & 3u), active, lane);
            float* rows = zs + (size_t)(t % 3u) * CL_SLOTS * ROW;
            float* sums = part + (size_t)(t & 1u) * CL_WARPS * CL_SLOTS * CPC;
            for (uint32_t first = 0; first < dp.n; first += CL_SLOTS) {
                const int n = (int)min((uint32_t)CL_SLOTS, dp.n - first);
                if (first) {
                    cl_bar_contract();
                    for (int s = warp; s < n; s += CL_WARPS) {
                        const uint4 rec = __ldcg(reinterpret_cast<const uint4*>(&c.cell_sorted[dp.begin + first + s]));
                        if (rec.x < c.frame_cap)
                            for (int p = lane; p < H / 4; p += 32)
                                *reinterpret_cast<float4*>(rows + (size_t)s * ROW + 4 * p) = ldcg4(c.dhp + (size_t)rec.x * H + 4 * p);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    cl_bar_contract();
                }
                cl_contract<CPC, KPT>(w, rows + k0, ROW, n, sums + (size_t)warp * CL_SLOTS * CPC, lane);
                cl_bar_contract();
                if (first + CL_SLOTS >= dp.n && warp == CL_WARPS - 1) cl_arrive_all(read0 + 8 * (t & 3u), active, lane);
                // a warp finishes 32 columns of a cell at a time
                for (int item = warp; item < n * FC; item += CL_WARPS) {
                    const int cell_i = item / FC, f = item % FC;
                    const uint4 rec = first ? __ldcg(reinterpret_cast<const uint4*>(&c.cell_sorted[dp.begin + first + cell_i])) : R.rec[t % CL_RING][cell_i];
                    const uint4 link = first ? __ldcg(&c.cell_link[dp.begin + first + cell_i]) : R.link[t % CL_RING][cell_i];
                    const int jj = 32 * f + lane, col = j0 + jj, cc = col < H ? col : col - H;
                    const uint32_t ch = col < H ? rec.y : rec.z, lk = col < H ? link.x : link.y;
                    const bool live = jj < CPC && col < K2 && rec.x < c.frame_cap && ch < c.frame_cap, cell = live && !(lk >> 31);
                    float v = 0.f;
                    if (live) {
                        float hv;
                        float4 a, b;
                        if (first == 0) {
                            hv = hs[((size_t)(t % 4u) * CL_SLOTS + cell_i) * CPC + jj];
                            const float4* d4 = reinterpret_cast<const float4*>(dls + (((size_t)(t % 4u) * CL_SLOTS + cell_i) * 2 + (col < H ? 0 : 1)) * 8);
                            a = d4[0]; b = d4[1];
                        } else {
                            hv = __ldcg(&c.arena[(size_t)ch * H + cc]);
                            a = ldcg4(c.dlog + (size_t)ch * 8); b = ldcg4(c.dlog + (size_t)ch * 8 + 4);
                        }
                        v = cl_total<CPC>(sums, cell_i, jj);
                        const float* wf = ws + jj;
                        v = fmaf(wf[0], a.x, v); v = fmaf(wf[CPC], a.y, v); v = fmaf(wf[2 * CPC], a.z, v); v = fmaf(wf[3 * CPC], a.w, v);
                        v = fmaf(wf[4 * CPC], b.x, v); v = fmaf(wf[5 * CPC], b.y, v); v = fmaf(wf[6 * CPC], b.z, v); v = fmaf(wf[7 * CPC], b.w, v);
                        if (cell) v *= 1.f - hv * hv;
                    }
                    if (t > 1 && first == 0) mbar_wait(c, read0 + 8 * ((t - 2u) & 3u), ((t - 2u) >> 2) & 1u);
                    // (row of the callee: the columns of every 16-byte piece belong to one callee)
                    const uint32_t base = smem_u32(zs + (size_t)((t + 1u) % 3u) * CL_SLOTS * ROW) - (col < H ? 0u : 4u * H);
                    cl_push_row<(CPC < 32 ? CPC : 32)>(v, cell && lk < (uint32_t)CL_SLOTS && t + 1u < steps, base + 4u * (lk * ROW),
                                                       4u * (j0 + 32 * f), full0 + 8 * ((t + 1u) % 3u), active, lane);
                    if (cell) c.dhp[(size_t)ch * H + cc] = v;
                    else if (live && (lk & 0x7FFFFFFFu) < (uint32_t)c.V) atomicAdd(c.dE + (size_t)(lk & 0x7FFFFFFFu) * c.D + cc, v);
                }
            }
            __syncwarp();
        }
        if (t + 1u < steps && R.depth[(t + 1u) % CL_RING].n > (uint32_t)CL_SLOTS) {
            cluster_sync_all();
        }
    }
    cluster_sync_all();
    if (blockIdx.x == 0 && threadIdx.x == 0) c.ctl->waves_backward += top - d0;      // (after the grid-wide kernel's count)
}

template <int CPC, int KPT>
constexpr size_t cl_smem_bytes(bool gradient) {
    const size_t row = (size_t)CL_WARPS * (CPC < 32 ? 2 : 1) * KPT;
    return (3 * CL_SLOTS * row + 2 * (size_t)CL_WARPS * CL_SLOTS * CPC + (gradient ? 4 * CL_SLOTS * (CPC + 16) + 8 * CPC : 0)) * sizeof(float);
}
