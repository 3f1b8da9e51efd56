// Scheduling of structural recursion over the input trees:
//
//     f(v) = leaf(tok v)                      if is_leaf(v)
//          = cell(f(child v), f(child v))     otherwise            (optionally under the per-node loss)
//
// Every Call_i of such a program is decided by the input structure alone, and the two operands of a cell are the results
// of the two calls its own invocation made: when the calls fire, the frames whose states the match will bring together are
// known.  So one pass down the recursion -- level by level, all instances at once -- makes the frames (tags), the operand
// references of every cell and all lists the later kernels read; no token travels back up and no match is looked up.  The
// general scheduler (rdf_scheduler_kernel) needs a second wave per level for the returning tokens, and its interpreter a
// dozen dependent steps per token.
//
// What bounds it is the latency of a level: the level's records (L2), the words of the children (L2 or DRAM), one barrier.
// Measured, general scheduler with its list kernels -> this kernel: 8192 sentence trees (320 638 invocations, 16 levels)
// 0.338 -> 0.072 ms; 48 trees 0.149 -> 0.021 ms; 64 chains of depth 4096 with 16 perfect trees 21.1 -> 4.2 ms.
//
// Places are handed out by prefix sums, not by counters: the thread that creates a child sees whether it is a cell, so the
// cells of the next level are counted per chunk of FS_CHUNK records while the level is written, and after the barrier
// every block adds up the counts of the chunks before its own.  Frame ids, list positions and operand rows are therefore
// a function of the input alone (breadth first, instances in order): sums over the lists have the same order on every run.
// (Included by rdf_exec.cu only: it defines kernels.)
#pragma once
#include "rdf_exec.h"

static const int FS_CHUNK = 512;               // threads per block = records per chunk
static const uint32_t FS_ONE_BLOCK = 4096;     // runs with at most this many frames: one block
static const uint32_t FS_STRETCH = 4096;       // narrow levels block 0 runs alone before it meets the grid again

struct FoldShared {
    uint4    q[2][FS_CHUNK];                   // records of a narrow level, by level parity
    uint32_t wcell[2][FS_CHUNK / 32], wbelow[FS_CHUNK / 32], wall[FS_CHUNK / 32];
};

// where a level lies: n records whose frames are [fb, fb + n); cb / lb cells and leaves in the levels above
struct FoldLevel {
    uint32_t n, fb, cb, lb, d;
};

// The words of node v: left, right, token.  (A bad index is caught by fold_record; the loads of several nodes are issued
// before the first of them is looked at.)
// AHEAD: the sector 128 bytes on is fetched to L1 meanwhile (by the nodes at the start of a sector).  The nodes of a tree are
// usually stored in the order of the descent, so that is where the next levels of a thin recursion look.
struct NodeWords {
    int32_t l, r, t;
    bool in;
};
template <bool AHEAD>
__device__ __forceinline__ NodeWords fold_words(const DevCtx& c, int32_t v) {
    NodeWords w;
    w.in = v >= 0 && v < c.N;
    w.l = -1; w.r = 0; w.t = -1;
    if (w.in) {
        w.l = __ldg(&c.left[v]); w.r = __ldg(&c.right[v]); w.t = __ldg(&c.tok[v]);
        if (AHEAD && (v & 7) < 2 && v + 32 < c.N) {
            asm volatile("prefetch.global.L1 [%0];" ::"l"(c.left + v + 32));
            asm volatile("prefetch.global.L1 [%0];" ::"l"(c.right + v + 32));
            asm volatile("prefetch.global.L1 [%0];" ::"l"(c.tok + v + 32));
        }
    }
    return w;
}
// The record of a node: {left, right or token, instance, -}; left < 0: a leaf.  A node outside the arrays or a leaf whose
// token is no row of the embedding table is reported, and stands for a leaf of token 0.
__device__ __forceinline__ uint4 fold_record(const DevCtx& c, const NodeWords& w, uint32_t inst) {
    if (!w.in || (w.l < 0 && (w.t < 0 || w.t >= c.V))) {
        set_status(c, RDF_ERR_BAD_ARG);
        return make_uint4(0xFFFFFFFFu, 0u, inst, 0u);
    }
    return make_uint4((uint32_t)w.l, (uint32_t)(w.l < 0 ? w.t : w.r), inst, 0u);
}
__device__ __forceinline__ void fold_frame(const DevCtx& c, uint32_t id, uint32_t parent, uint32_t label, uint32_t wave, int32_t node, uint32_t inst) {
    Frame f;
    f.parent = parent; f.label = label | (wave << FRAME_WAVE_SHIFT); f.arg = node;
    c.frames[id] = f;
    if (c.finst) c.finst[id] = inst;
}

// instance b: the context of `result` and the invocation it calls
__device__ __forceinline__ uint4 fold_seed(const DevCtx& c, uint32_t b) {
    const int32_t root = __ldg(&c.tree_root[b]);
    const uint32_t id = (uint32_t)c.B + b;
    Frame f;
    f.parent = LEAF_MARK; f.label = 0; f.arg = root;
    c.frames[b] = f;
    fold_frame(c, id, b, (uint32_t)c.fold_label[2], 0u, root, b);
    if (c.finst) c.finst[b] = b;
    if (c.zdst) c.zdst[id] = NO_ZDST;
    c.y[b] = id;
    return fold_record(c, fold_words<false>(c, root), b);
}

// One record of a level: its operator goes to the lists; a cell makes its two calls.  next: where the records of the next
// level go; counts: the counters of its chunks (null: a next level that one block runs alone).  Called by whole warps.
__device__ __forceinline__ void fold_fire(const DevCtx& c, const FoldLevel& L, uint32_t p, bool valid, const uint4& rec, const int32_t (&arg)[2],
                                          const uint4 (&kid)[2], uint32_t rank, uint4* next, uint32_t* counts) {
    const uint32_t f = L.fb + p;
    const bool cell = valid && (int32_t)rec.x >= 0;
    if (cell) {
        const uint32_t pos = L.cb + rank, k0 = L.fb + L.n + 2u * rank, k1 = k0 + 1u;
        c.op_l[f] = k0; c.op_r[f] = k1;
        c.all_cells[pos] = f;
        c.cell_ops[pos] = make_uint4(f, k0, k1, 1u);
        if (c.cell_pos) c.cell_pos[f] = pos;
        if (c.zdst) *reinterpret_cast<uint2*>(&c.zdst[k0]) = make_uint2(2u * pos, 2u * pos + 1u);
        fold_frame(c, k0, f, (uint32_t)c.fold_label[0], L.d + 1u, arg[0], rec.z);
        fold_frame(c, k1, f, (uint32_t)c.fold_label[1], L.d + 1u, arg[1], rec.z);
        next[2u * rank] = kid[0];
        next[2u * rank + 1u] = kid[1];
    } else if (valid) {
        const uint32_t pos = L.lb + p - rank;
        c.op_l[f] = LEAF_MARK; c.op_r[f] = rec.y;
        LeafItem it;
        it.slot = f; it.tok = (int32_t)rec.y;
        c.leaf_items[pos] = it;
        if (c.lstm) {
            c.all_leaves[pos] = f;
            if (c.cell_pos) c.cell_pos[f] = pos;
            if (c.leaf_ops) c.leaf_ops[pos] = make_uint4(f, rec.y, 0u, 1u);
        }
    }
    if (counts) {
        // the cells among the warp's new records, per chunk (the warp's cells have consecutive ranks: two chunks at most)
        const unsigned cells = __ballot_sync(0xffffffffu, cell);
        if (cells) {
            const uint32_t first = __shfl_sync(0xffffffffu, rank, __ffs(cells) - 1) / (FS_CHUNK / 2);
            const unsigned a = __ballot_sync(0xffffffffu, cell && (int32_t)kid[0].x >= 0), b = __ballot_sync(0xffffffffu, cell && (int32_t)kid[1].x >= 0);
            const unsigned here = __ballot_sync(0xffffffffu, cell && rank / (FS_CHUNK / 2) == first);
            if (threadIdx.x % 32 == 0) {
                const uint32_t n0 = __popc(a & here) + __popc(b & here), n1 = __popc(a & ~here) + __popc(b & ~here);
                if (n0) atomicAdd(&counts[first], n0);
                if (n1) atomicAdd(&counts[first + 1u], n1);
            }
        }
    }
}

// what the record's thread needs of its children: fetched before the places are known
template <bool AHEAD>
__device__ __forceinline__ void fold_children(const DevCtx& c, const uint4& rec, bool cell, int32_t (&arg)[2], uint4 (&kid)[2]) {
    arg[0] = arg[1] = 0;
    kid[0] = kid[1] = make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
    if (cell) {
        arg[0] = (int32_t)(c.fold_right[0] ? rec.y : rec.x);
        arg[1] = (int32_t)(c.fold_right[1] ? rec.y : rec.x);
        const NodeWords a = fold_words<AHEAD>(c, arg[0]), b = fold_words<AHEAD>(c, arg[1]);
        kid[0] = fold_record(c, a, rec.z);
        kid[1] = fold_record(c, b, rec.z);
    }
}

// Room for the next level?  The same answer in every block.
__device__ __forceinline__ bool fold_room(const DevCtx& c, const FoldLevel& L, uint32_t cells) {
    const uint64_t end = (uint64_t)L.fb + L.n + 2ull * cells;
    if (end > c.frame_cap) { set_status(c, RDF_ERR_FRAMES_FULL); return false; }
    if (2ull * cells > c.qcap) { set_status(c, RDF_ERR_QUEUE_FULL); return false; }      // (the records of the level would not fit)
    // (in token waves a level costs one on the way down and one on the way up)
    if (cells && 2ull * (L.d + 1u) + 3u > c.wave_limit) { set_status(c, RDF_ERR_WAVE_LIMIT); return false; }
    return true;
}

__device__ __forceinline__ void fold_next(const DevCtx& c, FoldLevel& L, uint32_t cells) {
    if (blockIdx.x == 0 && threadIdx.x == 0 && L.d < c.wave_cap)
        c.wave_marks[L.d] = make_uint4(L.fb, L.fb + L.n, L.cb, L.cb + cells);
    L.fb += L.n;
    L.cb += cells;
    L.lb += L.n - cells;
    L.n = 2u * cells;
    ++L.d;
}

__global__ void __launch_bounds__(FS_CHUNK, 1) rdf_fold_kernel(const __grid_constant__ DevCtx c) {
    __shared__ FoldShared sh;
    const uint32_t tid = threadIdx.x, lane = tid % 32, warp = tid / 32, B = (uint32_t)c.B;
    uint4* const tq[2] = {reinterpret_cast<uint4*>(c.q[0]), reinterpret_cast<uint4*>(c.q[1])};
    FoldLevel L{B, B, 0u, 0u, 0u};
    uint32_t generation = 0, g = 0, stretch = 0;
    const long long t_start = clock64();
    bool in_shared = false, alive = true;
    if (3ull > c.wave_limit) { set_status(c, RDF_ERR_WAVE_LIMIT); alive = false; }
    else if (2ull * B > c.frame_cap) { set_status(c, RDF_ERR_FRAMES_FULL); alive = false; }
    else if (B <= FS_CHUNK) {
        // few instances: block 0 starts alone
        if (blockIdx.x == 0 && tid < B) sh.q[0][tid] = fold_seed(c, tid);
        __syncthreads();
        in_shared = true;
    } else {
        const uint32_t chunks = (B + FS_CHUNK - 1) / FS_CHUNK;
        for (uint32_t k = blockIdx.x; k < chunks; k += gridDim.x) {
            const uint32_t b = k * FS_CHUNK + tid;
            bool cell = false;
            if (b < B) {
                const uint4 rec = fold_seed(c, b);
                tq[0][b] = rec;
                cell = (int32_t)rec.x >= 0;
            }
            const unsigned m = __ballot_sync(0xffffffffu, cell);
            if (lane == 0 && m) atomicAdd(&c.level_counts[k], (uint32_t)__popc(m));
        }
        alive = grid_barrier(c, &c.ctl->bar.v, generation);
    }
    while (alive && L.n) {
        if (L.n <= FS_CHUNK) {
            // A narrow level fits one block: block 0 runs level after level out of its shared memory with block barriers while
            // the others wait at the grid barrier, until a level is wider (or FS_STRETCH levels, so that no wait expires).
            if (blockIdx.x == 0) {
                uint32_t k = 0;
                do {
                    const bool valid = tid < L.n;
                    uint4 rec = make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
                    if (valid) rec = in_shared ? sh.q[L.d & 1][tid] : __ldcg(&tq[L.d & 1][tid]);
                    const bool cell = valid && (int32_t)rec.x >= 0;
                    int32_t arg[2];
                    uint4 kid[2];
                    fold_children<true>(c, rec, cell, arg, kid);
                    const unsigned m = __ballot_sync(0xffffffffu, cell);
                    if (lane == 0) sh.wcell[L.d & 1][warp] = __popc(m);
                    __syncthreads();
                    const uint32_t w = lane < FS_CHUNK / 32 ? sh.wcell[L.d & 1][lane] : 0u;
                    const uint32_t total = __reduce_add_sync(0xffffffffu, w);
                    const uint32_t rank = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) + __popc(m & ((1u << lane) - 1u));
                    if (!fold_room(c, L, total)) { L.n = 0; break; }
                    const bool stay = 2u * total <= FS_CHUNK;
                    if (warp * 32u < L.n)
                        fold_fire(c, L, tid, valid, rec, arg, kid, rank, stay ? sh.q[(L.d + 1) & 1] : tq[(L.d + 1) & 1],
                                  stay ? nullptr : c.level_counts + (g % 3u) * c.level_cap);
                    fold_next(c, L, total);
                    in_shared = stay;
                    __syncthreads();
                } while (L.n && L.n <= FS_CHUNK && ++k < FS_STRETCH);
                if (in_shared && tid < L.n) tq[L.d & 1][tid] = sh.q[L.d & 1][tid];       // (a stretch that was cut short)
                in_shared = false;
                if (tid == 0) {
                    uint4* s = &c.ctl->fold_state[2 * (stretch & 1u)];
                    s[0] = make_uint4(L.n, L.fb, L.cb, L.lb);
                    s[1] = make_uint4(L.d, 0u, 0u, 0u);
                }
            }
            if (gridDim.x > 1 && !grid_barrier(c, &c.ctl->bar.v, generation)) { alive = false; break; }
            const uint4* s = &c.ctl->fold_state[2 * (stretch & 1u)];     // (two slots in turn: block 0 may be a stretch ahead)
            if (blockIdx.x != 0) {
                const uint4 a = __ldcg(s), b = __ldcg(s + 1);
                L.n = a.x; L.fb = a.y; L.cb = a.z; L.lb = a.w; L.d = b.x;
            }
            in_shared = false;
            ++stretch;
            continue;
        }
        // ---- a wide level: the chunks in contiguous ranges, one per block
        const uint32_t chunks = (L.n + FS_CHUNK - 1) / FS_CHUNK, per = (chunks + gridDim.x - 1) / gridDim.x;
        const uint32_t k0 = min(chunks, blockIdx.x * per), k1 = min(chunks, k0 + per);
        const uint4* q = tq[L.d & 1];
        uint32_t* counts = c.level_counts + (g % 3u) * c.level_cap;
        uint32_t p = k0 * FS_CHUNK + tid;
        uint4 rec = make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
        if (k0 < k1 && p < L.n) rec = __ldcg(&q[p]);
        uint32_t below = 0, all = 0;
        for (uint32_t k = tid; k < chunks; k += FS_CHUNK) {
            const uint32_t v = __ldcg(&counts[k]);
            all += v;
            if (k < k0) below += v;
        }
        // (the counters of the level before are free: zero for the level after the next)
        {
            uint32_t* old = c.level_counts + ((g + 2u) % 3u) * c.level_cap;
            for (uint32_t k = blockIdx.x * FS_CHUNK + tid; k < c.level_cap; k += gridDim.x * FS_CHUNK) old[k] = 0u;
        }
        uint32_t base = 0, total = 0;
        bool room = true;
        for (uint32_t k = k0; k == k0 || k < k1; ++k) {
            const bool valid = k < k1 && p < L.n, cell = valid && (int32_t)rec.x >= 0;
            int32_t arg[2];
            uint4 kid[2];
            fold_children<false>(c, rec, cell, arg, kid);
            const uint4 cur = rec;
            if (k == k0) {
                below = __reduce_add_sync(0xffffffffu, below);
                all = __reduce_add_sync(0xffffffffu, all);
                if (lane == 0) { sh.wbelow[warp] = below; sh.wall[warp] = all; }
            }
            if (k + 1 < k1 && p + FS_CHUNK < L.n) rec = __ldcg(&q[p + FS_CHUNK]);          // in flight during this chunk
            const unsigned m = __ballot_sync(0xffffffffu, cell);
            if (lane == 0) sh.wcell[k & 1][warp] = __popc(m);
            __syncthreads();
            if (k == k0) {
                base = __reduce_add_sync(0xffffffffu, lane < FS_CHUNK / 32 ? sh.wbelow[lane] : 0u);
                total = __reduce_add_sync(0xffffffffu, lane < FS_CHUNK / 32 ? sh.wall[lane] : 0u);
                room = fold_room(c, L, total);
                if (!room) break;
            }
            const uint32_t w = lane < FS_CHUNK / 32 ? sh.wcell[k & 1][lane] : 0u;
            const uint32_t rank = base + __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) + __popc(m & ((1u << lane) - 1u));
            base += __reduce_add_sync(0xffffffffu, w);
            fold_fire(c, L, p, valid, cur, arg, kid, rank, tq[(L.d + 1) & 1],
                      2u * total > FS_CHUNK ? c.level_counts + ((g + 1u) % 3u) * c.level_cap : nullptr);
            p += FS_CHUNK;
        }
        if (!room) { alive = false; break; }
        fold_next(c, L, total);
        ++g;
        if (gridDim.x > 1) alive = grid_barrier(c, &c.ctl->bar.v, generation);
        else __syncthreads();
    }
    // every block knows the totals: the rows after the last cell, which the weight gradient reads in whole stages, are zero
    if (alive && blockIdx.x == gridDim.x - 1) zero_tail_rows(c, L.cb, L.lb);
    if (blockIdx.x == 0 && tid == 0) {
        const uint32_t inv = L.cb + L.lb;
        c.ctl->frame_count.v = B + inv; c.ctl->cell_count.v = L.cb; c.ctl->leaf_count.v = L.lb;
        c.ctl->all_cells = L.cb; c.ctl->all_leaves = L.lb;
        c.ctl->n_depth_waves = min(L.d, c.wave_cap);
        c.ctl->call_waves = L.d;
        // in terms of the token waves of the graph: a call per invocation, a return per invocation, one more for `result`
        c.ctl->waves = 2u * L.d + 1u;
        // (the widest wave: its calls and returns belong to invocations none of which is below another one, and no such set
        // is larger than that of the leaves)
        c.ctl->max_wave_tokens = max(B, L.lb);
        c.ctl->invocations = inv; c.ctl->tokens = (unsigned long long)B + 2ull * inv;
        c.ctl->store_inserts = c.ctl->store_matches = c.ctl->cells = L.cb;
        c.ctl->leaves = L.lb;
        c.ctl->cyc[0] = clock64() - t_start;
        c.ctl->forward_status = ld_volatile_i32(&c.ctl->status);
    }
}
