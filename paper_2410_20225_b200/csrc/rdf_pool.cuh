// Integer programs run out of shared memory: one pool of tokens per thread block.
//
// Tokens of different instances never meet, and inside an instance only the frames of the calls in flight are needed: a
// block takes instances, keeps their frames, pending tokens and parked operands in its shared memory, and works depth-first
// -- in rounds of up to one token per thread from the top of a stack -- until they have returned their results; then it
// takes more.  Nothing of a call goes to global memory but its argument and its result.  (The general scheduler runs all
// instances in step, breadth-first: its queues, frames and store hold a whole wave, so every token costs about 128 bytes and
// three or four dependent L2 round trips, and every wave a grid barrier.)
//
// A token is a frame that waits to be entered, or a frame whose match node has all its operands and waits to go on; the two
// kinds have a stack each.  A round: the warps take completed matches first (they give frames back) and the other warps the
// top of the frames to enter, so that the threads of a warp do the same thing.  A thread runs one segment: new frames for
// the calls it makes, pushed as tokens; or a value that is returned -- parked in the caller's frame, and if it was the last
// operand the match becomes a token (carrying on in the same thread instead leaves the warp to a few long chains of returns:
// 131 072 calls of fib took 13.0 ms with up to three in a row, 24.7 with eight, 7.8 with none, before the other measures).
// The program is a fused form of the lowered code (PoolBuilder): operands are register + immediate, a comparison branches by
// itself, consecutive calls reserve their frames together.
//
// Segments of the common shapes (a list of conditions that ends in a return or in calls; an operator and a return; a tail
// call) run without the interpreter, from registers.
//
// What bounds it: the latency of a round -- some 400 dependent instructions per warp between two block barriers -- and the
// frames that fit the shared memory, which limit the tokens of a round.  (16 384 calls of fib(0..18): an instruction issued in
// 55 % of the cycles, 19.3 warp instructions per call; warps stalled per issue: 2.6 on the fixed latency of the instruction
// before, 2.2 at the barrier, 1.9 on shared memory.)
// Measured, general scheduler -> this: 131 072 calls of fib(0..18) 36.3 -> 5.3 ms, 1024 calls 0.72 -> 0.18 ms, 8 calls of
// fib(0..10) 0.137 -> 0.037 ms, 200 calls of tak 1.75 -> 0.80 ms (limited by the depth of the largest instance).
// Handing calls of a busy block to idle ones through global memory was built and dropped: 200 calls of tak 0.90 -> 0.83 ms,
// but 1024 calls of fib 0.23 -> 0.31 ms.
// Programs of one function whose calls meet in one operator (fib and tak among them) have an executor of their own, without rounds
// (rdf_lanes.cuh); the figures here are from before it.
// (Included by rdf_exec.cu only: it defines kernels.)
#pragma once
#include "rdf_exec.h"

static const int POOL_THREADS = 768, POOL_PER_SM = 1;   // threads of a block, blocks per SM (131 072 calls of fib: 512 threads 6.7 ms, 768 5.5,
                                                        // 1024 6.2, two blocks of 256 6.7: more threads leave each fewer frames)
// A block runs its instances to their end, and an instance far larger than the others would keep one block busy long after the
// device has run out of work (one of fib(30), 2.7 M calls, 22.9 ms).  When at most POOL_ACTIVE blocks are left, one with more
// tokens pending than threads all the while leaves them to the general scheduler, which spreads a wave over the device: its
// frames, parked operands and the calls to be entered go there as they are.  Before that it runs as long as the other way
// costs: some 20 us to get going, and the clearing of the token store (PoolSizes::hand_after).
static const uint32_t POOL_ACTIVE = 8;
static const uint32_t POOL_ROOT = 0x80000000u;          // frame word of an instance's `result` context: | instance
// Frame word of an invocation: parent frame [15:0], label [21:16], depth of the tag [27:22] (path tags)

struct PoolSizes {
    uint32_t cap;            // frames of a block
    uint32_t div_shift, reserve;   // pool_width
    uint32_t cont_calls;     // a completed match may take frames too
    uint32_t chunk;          // instances a block takes at a time
    uint32_t refill;         // it takes them when fewer tokens than this are pending
    uint32_t max_depth;      // path tags: labels that fit the packed tag; frame tags: no limit (0xFFFFFFFF)
    unsigned long long max_calls;   // frame tags: Call firings the caller allows
    unsigned long long max_parked;  // path tags: operands the token store of the call holds
    uint32_t n_match;        // match nodes, at least 1
    int      match_step;     // -1, 1: direction in which Pool::match grows
    uint32_t hand_slots;     // places for the frames of a block that leaves its calls to the general scheduler
    long long hand_after;    // clock cycles it runs on its own before it does
    uint32_t late_waves;     // PoolThread::n_late
    int      fallback;       // the general scheduler is launched behind this kernel for a pool that is exhausted
};

static const int POOL_LEAVE = 3;
struct PoolShared {
    uint32_t entered[2];     // frames to enter pushed in the round (by parity)
    uint32_t matched[2];     // completed matches pushed in the round
    uint32_t taken[2];       // frames taken in the round
    uint32_t freed[2];       // frames given back in the round
    uint32_t next_chunk;
    uint32_t waves[POOL_BINS];   // tokens per wave (of the block), the first POOL_BINS waves
    uint32_t hand;           // 1 + the place the block leaves its frames in
    uint32_t left[3];        // of a block that leaves them: first free frame, free frames, frames to enter
    long long alone;         // since when few others are left (clock cycles; 0: they are not)
    int      stop;           // 1: an error, 2: the pool is exhausted, POOL_LEAVE: the block leaves its calls
};

inline size_t pool_fixed_bytes(const PoolProgram& P) { return sizeof(PoolProgram) + (size_t)(P.n_regs + 1) * POOL_THREADS * 8; }
__host__ __device__ inline bool pool_tokens_share(const PoolProgram& P) { return P.n_match <= 1; }       // one token per frame at most: Pool::match
inline size_t pool_frame_bytes(const PoolProgram& P) {
    return 8 * (size_t)P.words + 4 + 4 * (size_t)std::max(1, P.n_match) + 2 + 2 + (pool_tokens_share(P) ? 0 : 2);
}
static const uint32_t POOL_MAX_FRAMES = 1u << 13;       // a completed match: frame | node << 13

// The pool's arrays in dynamic shared memory
struct Pool {
    const PoolProgram* prog;
    int64_t*  regs;          // [n_regs + 1][T]; the last one is zero
    int64_t*  words;         // [words][cap]: arguments while the frame waits to be entered, then the operands of its match nodes
    uint32_t* head;          // [cap] frame word
    uint32_t* state;         // [n_match][cap] waiting to be entered (the first row): its wave; then per match node the operands that
                             // have arrived [7:0] and the latest wave one of them arrived in [31:8]
    uint16_t* enter;         // [cap] frames to enter, oldest first (a deque)
    uint16_t* match;         // stack of completed matches; one match node (a frame has one token then): it grows down from the end of
                             // `enter`, more of them: an array of its own
    uint16_t* ring;          // [cap] free frames, oldest first
};

// a place on a shared counter for every thread that gets here together: one atomic per group
__device__ __forceinline__ uint32_t pool_take(uint32_t* counter) {
    const uint32_t group = __activemask(), lane = threadIdx.x & 31u, leader = __ffs(group) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(counter, (uint32_t)__popc(group));
    return __shfl_sync(group, base, leader) + __popc(group & ((1u << lane) - 1u));
}

static const int POOL_RUN_BITS = 6;                     // calls that follow one another: at most POOL_MAX_CODE
static_assert(POOL_MAX_CODE < (1 << POOL_RUN_BITS), "a run of calls fits the bits of reserve");

// A block's frames on their way to the general scheduler, in the second wave queue
struct PoolDump {
    int64_t  *words;
    uint32_t *head, *state, *id;                // id: frame id, ~0: no frame; state ~0: to be entered
    __device__ PoolDump(const DevCtx& c, uint32_t slot) {
        char* p = reinterpret_cast<char*>(c.q[1]) + slot * c.pool.slot_bytes;
        words = reinterpret_cast<int64_t*>(p);
        head = reinterpret_cast<uint32_t*>(words + (size_t)c.pool.words * c.pool.cap);
        state = head + c.pool.cap;
        id = state + (size_t)c.pool.n_match * c.pool.cap;
    }
};
inline size_t pool_dump_bytes(const PoolProgram& P, uint32_t cap) { return (size_t)cap * (8 * (size_t)P.words + 8 + 4 * (size_t)std::max(1, P.n_match)); }

struct PoolThread {
    static const int T = POOL_THREADS;
    const DevCtx& c;
    const PoolSizes& z;
    const Pool& P;
    PoolShared& sh;
    uint32_t tid;
    uint32_t ring0, avail, ring_tail, enter0, match0, par;  // this round: first free frame, free frames, where frames go back, tops of the stacks
    uint32_t invocations = 0, inserts = 0, matches = 0, max_depth = 0, max_wave = 0;     // (max_wave: from POOL_BINS on)
    uint32_t* late_waves;    // tokens per wave from POOL_BINS on (global memory, n_late of them; later ones count in the last)
    uint32_t n_late;

    __device__ __forceinline__ int64_t val(uint32_t reg, int32_t imm) const { return P.regs[reg * T + tid] + (int64_t)imm; }
    __device__ __forceinline__ void set(uint32_t reg, int64_t v) { P.regs[reg * T + tid] = v; }
    __device__ __forceinline__ uint32_t wrap(uint32_t at) const { return at >= z.cap ? at - z.cap : at; }
    __device__ __forceinline__ void error(int code) {
        set_status(c, code);
        sh.stop = 1;
    }
    __device__ __forceinline__ void give_back(uint32_t f) { P.ring[wrap(ring_tail + pool_take(&sh.freed[par]))] = (uint16_t)f; }
    // k frames for calls that follow one another, and their places on the stack (first of each); false: the pool is exhausted.
    // The threads that get here together may make different numbers of calls (branches of a body, different functions): a
    // prefix sum over the lanes, one ballot per bit of k (k < 2^BITS).
    template <int BITS>
    __device__ __forceinline__ bool reserve(uint32_t k, uint32_t& frame_at, uint32_t& slot) {
        const uint32_t group = __activemask(), lane = threadIdx.x & 31u, leader = __ffs(group) - 1, lower = (1u << lane) - 1u;
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int b = 0; b < BITS; ++b) {
            const uint32_t m = __ballot_sync(group, (k >> b) & 1u);
            before += (uint32_t)__popc(m & lower) << b;
            total += (uint32_t)__popc(m) << b;
        }
        uint32_t f0 = 0, s0 = 0;
        if (lane == leader) {
            f0 = atomicAdd(&sh.taken[par], total);
            s0 = atomicAdd(&sh.entered[par], total);
        }
        frame_at = __shfl_sync(group, f0, leader) + before;
        slot = __shfl_sync(group, s0, leader) + before;
        if (frame_at + k <= avail) return true;
        sh.stop = 2;
        return false;
    }

    // Waves.  The pool does not run in waves, but a token has one all the same -- that of the token that made its call, plus
    // one; a match fires in the latest wave one of its operands arrived in -- and what the general scheduler reports of its
    // waves (their number, the widest one) and refuses because of them is the same here.
    // A token of wave `wave` is taken.  (There are at most 2^24 waves: 24 bits wherever a wave is kept.)
    __device__ __forceinline__ bool count_wave(uint32_t wave) {
        if (wave < (uint32_t)POOL_BINS) {
            atomicAdd(&sh.waves[wave], 1u);
            return true;
        }
        if (wave >= c.wave_limit) {
            error(RDF_ERR_WAVE_LIMIT);
            return false;
        }
        max_wave = max(max_wave, wave);
        if (n_late) atomicAdd(&late_waves[min(wave - (uint32_t)POOL_BINS, n_late - 1u)], 1u);
        return true;
    }

    // The operand `v` arrives at port `port` of match node `node` in frame f; the last one makes the match a token.
    __device__ __forceinline__ void deliver(uint32_t f, uint32_t node, uint32_t port, int64_t v, uint32_t wave) {
        const PoolMatch M = P.prog->match[node];
        P.words[(M.word0 + port) * z.cap + f] = v;
        __threadfence_block();
        uint32_t* state = &P.state[node * z.cap + f];
        if (M.n_ports == 2) {                               // one exchange: the second operand gets the first one's word, and nobody follows
            const uint32_t mine = wave << 8 | 1u << port, there = atomicExch(state, mine);
            if (there == 0u) {
                ++inserts;
                return;
            }
            *state = max(there, mine) | M.all;
        } else {
            const uint32_t bit = 1u << port;
            uint32_t there = atomicCAS(state, 0u, wave << 8 | bit);
            while (there != 0u) {
                const uint32_t both = max(there & ~0xFFu, wave << 8) | (there & 0xFFu) | bit;
                if ((both & 0xFFu) == M.all) {              // (nobody follows the last one)
                    *state = both;
                    break;
                }
                const uint32_t seen = there;
                there = atomicCAS(state, seen, both);
                if (there == seen) there = 0u;
            }
            if (there == 0u) {
                ++inserts;
                return;
            }
        }
        ++matches;
        const uint32_t at = match0 + pool_take(&sh.matched[par]);
        if (at < z.cap) P.match[z.match_step * (int)at] = (uint16_t)(f | node << 13);
        else sh.stop = 2;                                   // (only bodies with several match nodes can have more matches than frames)
    }

    // a frame that waits to be entered
    __device__ __forceinline__ void fill_frame(uint32_t f, uint32_t n_args, int64_t a0, int64_t a1, int64_t a2, uint32_t head, uint32_t wave) {
        P.head[f] = head;
        P.words[f] = a0;
        if (n_args > 1) P.words[z.cap + f] = a1;
        if (n_args > 2) P.words[2 * z.cap + f] = a2;
        P.state[f] = wave;
    }
    // Call_i under the tag of frame word h: the depth of the new tag.  False (status set) when it does not fit.
    __device__ __forceinline__ bool push_tag(uint32_t h, uint32_t& depth) {
        depth = 0;
        if (z.max_depth == 0xFFFFFFFFu) return true;
        depth = ((h & POOL_ROOT) ? 0u : (h >> 22) & 63u) + 1u;
        if (depth > z.max_depth) {
            error(RDF_ERR_TAG_OVERFLOW);
            return false;
        }
        max_depth = max(max_depth, depth);
        return true;
    }
    // The call is frame f's own output and enters the same function: the callee takes over the frame (and returns to where its
    // caller would).
    __device__ __forceinline__ bool same_function(uint32_t h, uint32_t label) const {
        return !(h & POOL_ROOT) && P.prog->labels[(h >> 16) & 63u].entry == P.prog->labels[label].entry;
    }
    __device__ __forceinline__ void tail_call(uint32_t f, uint32_t h, uint32_t label, int64_t a0, int64_t a1, int64_t a2, uint32_t depth, uint32_t wave) {
        fill_frame(f, P.prog->labels[label].n_args, a0, a1, a2, (h & ~(63u << 22)) | depth << 22, wave);
        P.enter[wrap(enter0 + pool_take(&sh.entered[par]))] = (uint16_t)f;      // (one token per frame: the deque holds all frames)
    }
    __device__ __forceinline__ static int64_t pick(const PoolOperand& o, int64_t a0, int64_t a1, int64_t a2) {
        return (o.reg == 0 ? a0 : o.reg == 1 ? a1 : o.reg == 2 ? a2 : 0ll) + (int64_t)o.imm;
    }
    __device__ __forceinline__ static bool holds(int cmp, int64_t a, int64_t b) { return cmp == PC_LT ? a < b : (a == b) == (cmp == PC_EQ); }

    // Entering a function of the common shape.
    __device__ __forceinline__ int enter_fast(uint32_t& f, uint32_t& h, const PoolEntry& e, uint32_t wave) {
        const int64_t a0 = P.words[f], a1 = e.n_args > 1 ? P.words[z.cap + f] : 0ll, a2 = e.n_args > 2 ? P.words[2 * z.cap + f] : 0ll;
        int which = e.n_cond;
        if (e.n_cond > 1 && holds(e.cmp[1], pick(e.a[1], a0, a1, a2), pick(e.b[1], a0, a1, a2))) which = 1;
        if (e.n_cond > 0 && holds(e.cmp[0], pick(e.a[0], a0, a1, a2), pick(e.b[0], a0, a1, a2))) which = 0;
        const PoolAction& act = e.act[which];
        if (act.n_calls == 0) return give_value(f, h, pick(act.ops[0], a0, a1, a2), wave);
        const uint32_t k = act.n_calls;
        uint32_t depth, frame_at, slot;
        invocations += k;
        if (!push_tag(h, depth) || !reserve<2>(k, frame_at, slot)) return -1;      // (1 to 3 calls)
#pragma unroll
        for (uint32_t q = 0; q < 3; ++q)
            if (q < k) {
                const uint32_t nf = P.ring[wrap(ring0 + frame_at + q)], label = act.labels[q] & 0xFFu, n_args = act.labels[q] >> 8;
                P.enter[wrap(enter0 + slot + q)] = (uint16_t)nf;
                P.head[nf] = f | label << 16 | depth << 22;
                P.state[nf] = wave + 1u;
                P.words[nf] = pick(act.ops[3 * q], a0, a1, a2);
                if (n_args > 1) P.words[z.cap + nf] = pick(act.ops[3 * q + 1], a0, a1, a2);
                if (n_args > 2) P.words[2 * z.cap + nf] = pick(act.ops[3 * q + 2], a0, a1, a2);
            }
        return -1;
    }

    // Return_i: frame f (its word h) has the value v.  Returns the code to go on with (in frame f, r0 = v), or -1.
    __device__ __forceinline__ int give_value(uint32_t& f, uint32_t& h, int64_t v, uint32_t wave) {
        for (;;) {
            const PoolLabel L = P.prog->labels[(h >> 16) & 63u];
            give_back(f);
            f = h & 0xFFFFu;
            if (L.k_kind == K_PORT) {
                deliver(f, L.k_node, L.k_port, v, wave);
                return -1;
            }
            h = P.head[f];
            if (L.k_kind == K_SEG) {
                set(0, v);
                return L.k_pc;
            }                                               // (K_RET: the call was the caller's own output)
        }
    }

    // Token `f`: a frame to enter (node < 0), or the completed match `node` of frame f.
    __device__ __forceinline__ void run(uint32_t f, int node) {
        const PoolProgram& prog = *P.prog;
        uint32_t h = P.head[f], wave = 0;
        int pc;
        if (node >= 0) {
            const PoolMatch M = prog.match[node];
            wave = P.state[node * z.cap + f] >> 8;
            const int64_t* w = P.words + M.word0 * z.cap + f;
            const int64_t p0 = w[0], p1 = w[z.cap], p2 = M.n_ports > 2 ? w[2 * z.cap] : 0ll;
            const PoolCont& q = prog.cont_of[min(node, POOL_MAX_CONT - 1)];
            if (node < POOL_MAX_CONT && q.op == PI_CALL && same_function(h, q.label)) {
                uint32_t depth;
                ++invocations;
                if (push_tag(h, depth))
                    tail_call(f, h, q.label, pick(q.ops[0], p0, p1, p2), pick(q.ops[1], p0, p1, p2), pick(q.ops[2], p0, p1, p2), depth, wave + 1u);
                return;
            }
            if (node < POOL_MAX_CONT && q.op >= PI_ADD && q.op <= PI_MAX) {
                const int64_t a = pick(q.a, p0, p1, p2), b = pick(q.b, p0, p1, p2);
                const int64_t r = q.op == PI_ADD ? a + b : q.op == PI_SUB ? a - b : q.op == PI_MUL ? a * b : a > b ? a : b;
                pc = give_value(f, h, r + (int64_t)q.imm, wave);
                if (pc < 0) return;
            } else {
                set(0, p0); set(1, p1);
                for (uint32_t k = 2; k < M.n_ports; ++k) set(k, w[k * z.cap]);
                pc = M.cont;
            }
        } else {
            uint32_t n_args = 1;
            int fast = -1;
            pc = prog.result_entry;
            if (!(h & POOL_ROOT)) {
                const PoolLabel L = prog.labels[(h >> 16) & 63u];
                pc = L.entry;
                n_args = L.n_args;
                fast = L.fast;
            }
            wave = P.state[f];
            P.state[f] = 0u;
            for (uint32_t k = 1; k < z.n_match; ++k) P.state[k * z.cap + f] = 0u;
            if (!count_wave(wave)) return;
            if (fast >= 0) {
                pc = enter_fast(f, h, prog.entry_of[fast], wave);
                if (pc < 0) return;
            } else {
                set(0, P.words[f]);
                if (n_args > 1) set(1, P.words[z.cap + f]);
                if (n_args > 2) set(2, P.words[2 * z.cap + f]);
            }
        }
        uint32_t frame_at = 0, slot = 0, run_left = 0;
        for (uint32_t step = 0; step < (1u << 22); ++step) {
            const PoolInstr in = prog.code[pc++];
            const int64_t a = val(in.ra, in.ia);
            if (in.op == PI_BR) {                           // carry on when the comparison holds, else go to imm
                const int64_t b = val(in.rb, in.ib);
                if (!holds(in.cmp, a, b)) pc = in.imm;
            } else if (in.op == PI_RET) {
                pc = give_value(f, h, a, wave);
                if (pc < 0) return;
            } else if (in.op == PI_CALL) {
                const uint32_t label = (uint32_t)in.imm, n_args = prog.labels[label].n_args;
                uint32_t depth;
                ++invocations;
                if (!push_tag(h, depth)) return;
                const int64_t a1 = n_args > 1 ? val(in.rb, in.ib) : 0ll, a2 = n_args > 2 ? val(in.rc, in.ic) : 0ll;
                if (in.tail && same_function(h, label)) {
                    tail_call(f, h, label, a, a1, a2, depth, wave + 1u);
                    return;
                }
                if (run_left == 0) {
                    run_left = in.n_run;
                    if (!reserve<POOL_RUN_BITS>(run_left, frame_at, slot)) return;
                }
                --run_left;
                const uint32_t nf = P.ring[wrap(ring0 + frame_at++)];
                fill_frame(nf, n_args, a, a1, a2, f | label << 16 | depth << 22, wave + 1u);
                P.enter[wrap(enter0 + slot++)] = (uint16_t)nf;
                if (in.last) return;
            } else {
                const int64_t b = val(in.rb, in.ib);
                switch (in.op) {
                    case PI_ADD: set(in.dst, a + b); break;
                    case PI_SUB: set(in.dst, a - b); break;
                    case PI_MUL: set(in.dst, a * b); break;
                    case PI_MAX: set(in.dst, a > b ? a : b); break;
                    case PI_REM: set(in.dst, b == 0 ? 0 : a % b); break;
                    case PI_CMP: set(in.dst, holds(in.cmp, a, b)); break;
                    case PI_MOV: set(in.dst, a); break;
                    case PI_CONST: set(in.dst, prog.consts[in.imm]); break;
                    case PI_ARG: set(in.dst, P.words[in.imm * z.cap + f]); break;
                    case PI_JMP: pc = in.imm; break;
                    case PI_PORT:
                        deliver(f, in.imm, in.cmp, a, wave);
                        if (in.last) return;
                        break;
                    case PI_TREE: {
                        if (a < 0 || a >= c.N) {
                            error(RDF_ERR_BAD_ARG);
                            return;
                        }
                        const int32_t* src = in.cmp == PT_RIGHT ? c.right : in.cmp == PT_TOK ? c.tok : c.left;
                        const int32_t x = __ldg(&src[a]);
                        set(in.dst, in.cmp == PT_ISLEAF ? (int64_t)(x < 0) : (int64_t)x);
                        break;
                    }
                    case PI_OUT: {
                        const uint32_t inst = h & ~POOL_ROOT;
                        if (inst < c.B) c.y[inst] = a;
                        give_back(f);
                        return;
                    }
                    default: return;                        // PI_HALT
                }
            }
        }
        error(RDF_ERR_WAVE_LIMIT);
    }
};

// Frames a round may enter: one per thread while the pool has frames to spare for what they may call (2^div_shift each).  A reserve
// of (depth + 1) x (calls per body) frames stays untouched by rounds that enter two or more, so that a single frame at a
// time -- plain depth-first recursion -- always gets through where the depth is bounded.
__device__ __forceinline__ uint32_t pool_width(const PoolSizes& z, uint32_t avail) {
    return max(1u, avail > z.reserve ? (avail - z.reserve) >> z.div_shift : 0u);
}

__device__ __forceinline__ Pool pool_arrays(unsigned char* p, uint32_t cap, int n_regs, int words, uint32_t n_match, int match_step) {
    Pool P;
    P.prog = reinterpret_cast<const PoolProgram*>(p);
    p += sizeof(PoolProgram);
    P.regs = reinterpret_cast<int64_t*>(p); p += (size_t)(n_regs + 1) * POOL_THREADS * 8;
    P.words = reinterpret_cast<int64_t*>(p); p += (size_t)words * cap * 8;
    P.head = reinterpret_cast<uint32_t*>(p); p += (size_t)cap * 4;
    P.state = reinterpret_cast<uint32_t*>(p); p += (size_t)n_match * cap * 4;
    P.enter = reinterpret_cast<uint16_t*>(p); p += (size_t)cap * 2;
    if (match_step < 0) P.match = P.enter + cap - 1;
    else { P.match = reinterpret_cast<uint16_t*>(p); p += (size_t)cap * 2; }
    P.ring = reinterpret_cast<uint16_t*>(p);
    return P;
}

// The frames of a block that leaves its calls, as they lie.  (On its own: it takes everything from shared memory, so that the
// rounds keep nothing in registers for it.)
__device__ __noinline__ void pool_leave(const DevCtx& c, unsigned char* smem, const PoolShared& sh) {
    const PoolProgram& prog = *reinterpret_cast<const PoolProgram*>(smem);
    const uint32_t cap = c.pool.cap, slot = sh.hand - 1u, ring0 = sh.left[0], avail = sh.left[1], enter0 = 0u, ne = sh.left[2];
    const Pool P = pool_arrays(smem, cap, prog.n_regs, prog.words, c.pool.n_match, pool_tokens_share(prog) ? -1 : 1);
    constexpr uint32_t T = POOL_THREADS;
    uint8_t* kind = reinterpret_cast<uint8_t*>(P.regs);      // 0 free, 1 entered, 2 to be entered (18 KB and more, for 8192 frames at most)
    const uint32_t tid = threadIdx.x, n_match = c.pool.n_match;
    auto wrap = [&](uint32_t at) { return at >= cap ? at - cap : at; };
    for (uint32_t i = tid; i < cap; i += T) kind[i] = 1u;
    __syncthreads();
    for (uint32_t i = tid; i < avail; i += T) kind[P.ring[wrap(ring0 + i)]] = 0u;
    for (uint32_t i = tid; i < ne; i += T) kind[P.enter[wrap(enter0 + i)]] = 2u;
    __syncthreads();
    const PoolDump d(c, slot);
    for (uint32_t i = tid; i < cap; i += T) {
        const uint32_t head = P.head[i];
        uint32_t id = 0xFFFFFFFFu;
        if (kind[i]) id = head & POOL_ROOT ? head & ~POOL_ROOT : (uint32_t)c.B + aggregated_inc(&c.ctl->hand_frames);
        d.id[i] = id;
        d.head[i] = head;
        for (uint32_t k = 0; k < c.pool.words; ++k) d.words[(size_t)k * cap + i] = P.words[k * cap + i];
        for (uint32_t k = 0; k < n_match; ++k) d.state[(size_t)k * cap + i] = kind[i] == 2u ? 0xFFFFFFFFu : P.state[k * cap + i];
    }
    if (tid == 0) atomicOr(&c.ctl->hand_mask, 1u << slot);
}

// Every 32 rounds, one thread: has another block failed; does this one leave its calls?  pending: it has no more instances to start
// and more tokens than threads.  (On its own and seldom: the read of the other blocks' count takes a third of a round.)
__device__ __noinline__ void pool_look(const DevCtx& c, const PoolSizes& z, PoolShared& sh, bool pending) {
    if (ld_volatile_i32(&c.ctl->status) != 0) sh.stop = 1;
    if (!pending || z.hand_slots == 0u || sh.stop != 0) return;
    if (gridDim.x - ld_volatile_u32(&c.ctl->blocks_done.v) > POOL_ACTIVE) {
        sh.alone = 0ll;
        return;
    }
    const long long now = clock64();
    if (sh.alone == 0ll) sh.alone = now;
    else if (now - sh.alone >= z.hand_after) {
        const uint32_t slot = atomicAdd(&c.ctl->hand_claims, 1u);
        if (slot < z.hand_slots) {
            sh.hand = slot + 1u;
            atomicCAS(&sh.stop, 0, POOL_LEAVE);              // (unless the pool is exhausted in this very round)
        }
        sh.alone = now;
    }
}

// The end of a block that has run its instances: its waves, and (the block that ends last) the verdict on the capacities of the call.
// bins: tokens of the first POOL_BINS waves; max_wave: the thread's latest wave beyond them.
__device__ __forceinline__ void pool_report(const DevCtx& c, const uint32_t* bins, uint32_t max_wave, uint32_t n_late, unsigned long long max_calls,
                                            unsigned long long max_parked, int fallback, long long t_start, uint32_t* scratch) {
    const uint32_t tid = threadIdx.x, T = blockDim.x, *late_waves = reinterpret_cast<const uint32_t*>(c.q[0]);
    uint32_t w = max_wave;
    for (uint32_t i = tid; i < (uint32_t)POOL_BINS; i += T)
        if (bins[i]) {
            atomicAdd(&c.ctl->wave_tokens[i], bins[i]);
            w = max(w, i);
        }
    w = __reduce_max_sync(0xffffffffu, w);
    if ((tid & 31u) == 0 && (w || tid == 0)) atomicMax(&c.ctl->waves, w + 1u);
    if (blockIdx.x == 0 && tid == 0) c.ctl->cyc[0] = clock64() - t_start;
    __threadfence();
    __syncthreads();
    if (tid == 0) *scratch = atomicAdd(&c.ctl->blocks_done.v, 1u);
    __syncthreads();
    if (*scratch != gridDim.x - 1u) return;
    __threadfence();
    // the widest wave of the call
    uint32_t wide = 0, late = 0;
    const uint32_t n_waves = ld_volatile_u32(&c.ctl->waves);
    for (uint32_t i = tid; i < min(n_waves, (uint32_t)POOL_BINS); i += T) wide = max(wide, __ldcg(&c.ctl->wave_tokens[i]));
    if (n_waves > (uint32_t)POOL_BINS)
        for (uint32_t i = tid; i < min(n_waves - (uint32_t)POOL_BINS, n_late); i += T) {
            const uint32_t v = __ldcg(&late_waves[i]);
            (i + 1u < n_late ? wide : late) = max(v, i + 1u < n_late ? wide : late);
        }
    wide = __reduce_max_sync(0xffffffffu, wide);
    late = __reduce_max_sync(0xffffffffu, late);
    if ((tid & 31u) == 0) {
        atomicMax(&c.ctl->max_wave_tokens, max(wide, late));
        // (the last bin is a sum over waves, and an upper bound only)
        if (c.tag_mode == RDF_TAGS_PATH && wide > c.qcap && !c.ctl->pool_exhausted) set_status(c, RDF_ERR_QUEUE_FULL);
    }
    __syncthreads();
    if (tid == 0) {
        volatile Control* k = c.ctl;
        k->tokens = k->invocations + (unsigned long long)c.B;
        if (k->pool_exhausted) {
            if (!fallback) set_status(c, RDF_ERR_QUEUE_FULL);
        } else {
            if (c.tag_mode == RDF_TAGS_FRAME && k->invocations > max_calls) set_status(c, RDF_ERR_FRAMES_FULL);
            if (c.tag_mode == RDF_TAGS_PATH && k->store_inserts > max_parked) set_status(c, RDF_ERR_STORE_FULL);
        }
        k->forward_status = k->status;
    }
}

__global__ void __launch_bounds__(POOL_THREADS, POOL_PER_SM) rdf_pool_kernel(const __grid_constant__ DevCtx c, const __grid_constant__ PoolProgram program,
                                                                             const __grid_constant__ PoolSizes z) {
    constexpr uint32_t T = POOL_THREADS;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ PoolShared sh;
    const uint32_t tid = threadIdx.x;
    {
        uint32_t* dst = reinterpret_cast<uint32_t*>(smem);
        const uint32_t* src = reinterpret_cast<const uint32_t*>(&program);
        for (uint32_t i = tid; i < sizeof(PoolProgram) / 4; i += T) dst[i] = src[i];
    }
    const Pool P = pool_arrays(smem, z.cap, program.n_regs, program.words, z.n_match, z.match_step);
    for (uint32_t i = tid; i < z.cap; i += T) P.ring[i] = (uint16_t)i;
    P.regs[program.n_regs * T + tid] = 0ll;
    if (tid == 0) {
        sh.entered[0] = sh.entered[1] = sh.matched[0] = sh.matched[1] = sh.taken[0] = sh.taken[1] = sh.freed[0] = sh.freed[1] = 0u;
        sh.stop = 0; sh.hand = 0u; sh.alone = 0ll;
    }
    for (uint32_t i = tid; i < (uint32_t)POOL_BINS; i += T) sh.waves[i] = 0u;
    const long long t_start = clock64();
    const uint32_t B = (uint32_t)c.B, chunks = (B + z.chunk - 1) / z.chunk;
    uint32_t ib = min(B, blockIdx.x * z.chunk), ie = min(B, ib + z.chunk);       // instances this block has taken and not yet started
    bool more = blockIdx.x < chunks;
    PoolThread t{c, z, P, sh, tid};
    t.late_waves = reinterpret_cast<uint32_t*>(c.q[0]);
    t.n_late = z.late_waves;
    uint32_t ne = 0, nm = 0, ring0 = 0, avail = z.cap, par = 0;      // frames to enter, completed matches
    unsigned long long tokens = 0;
    bool leaving = false;
    __syncthreads();
    for (uint32_t round = 0;; ++round) {
        // ---- more instances, while few tokens are pending and at most half of the frames are in use
        if (more && ne + nm < z.refill && avail > z.cap / 2 && ib < ie) {
            const uint32_t k = min(min(ie - ib, T - min(ne, T)), avail / 4);
            if (tid < k) {
                const uint32_t f = P.ring[t.wrap(ring0 + tid)], inst = ib + tid;
                P.head[f] = POOL_ROOT | inst;
                P.words[f] = c.x ? c.x[inst] : (int64_t)c.tree_root[inst];
                P.state[f] = 0u;
                P.enter[t.wrap(ne + tid)] = (uint16_t)f;
            }
            ib += k; ne += k; avail -= k;
            ring0 = t.wrap(ring0 + k);
            if (ib == ie) {
                if (tid == 0) sh.next_chunk = gridDim.x + atomicAdd(&c.ctl->next_chunk, 1u);
                __syncthreads();
                const uint32_t q = sh.next_chunk;
                more = q < chunks;
                if (more) { ib = q * z.chunk; ie = min(B, ib + z.chunk); }
            }
            __syncthreads();
        }
        if (ne + nm == 0) {
            if (!more) break;
            if (avail > z.cap / 2) continue;
            if (tid == 0) sh.stop = 2;                       // (no token holds the missing frames: not a state this kernel gets into)
            __syncthreads();
            break;
        }
        // ---- this round's tokens: completed matches for the first warps, frames to enter for the others
        const uint32_t width = pool_width(z, avail);
        const uint32_t mm = min(min(nm, T), z.cont_calls ? width : T), w0 = (mm + 31u) & ~31u;
        const uint32_t me = leaving ? 0u : min(min(ne, T - w0), z.cont_calls && mm ? (width > mm ? width - mm : 0u) : width);
        uint32_t f = 0xFFFFFFFFu;
        int node = -1;
        if (tid < mm) {
            const uint32_t v = P.match[z.match_step * (int)(nm - 1u - tid)];
            f = v & (POOL_MAX_FRAMES - 1u);
            node = (int)(v >> 13);
        } else if (tid >= w0 && tid - w0 < me) f = P.enter[t.wrap(ne - 1u - (tid - w0))];
        tokens += mm + me;
        t.ring0 = ring0; t.avail = avail; t.ring_tail = t.wrap(ring0 + avail);
        t.enter0 = ne - me; t.match0 = nm - mm; t.par = par;
        __syncthreads();
        if (f != 0xFFFFFFFFu) t.run(f, node);
        if (tid == 0) {
            sh.entered[par ^ 1u] = 0u; sh.matched[par ^ 1u] = 0u; sh.freed[par ^ 1u] = 0u; sh.taken[par ^ 1u] = 0u;
            if ((round & 31u) == 31u) pool_look(c, z, sh, !more && ib >= ie && ne + nm >= T);
            if (c.tag_mode == RDF_TAGS_FRAME && tokens > 2ull * (z.max_calls + B) + T) {             // more calls than the caller allows
                set_status(c, RDF_ERR_FRAMES_FULL);
                sh.stop = 1;
            }
        }
        __syncthreads();
        ne = ne - me + sh.entered[par];
        nm = nm - mm + sh.matched[par];
        ring0 = t.wrap(ring0 + sh.taken[par]);
        avail = avail - sh.taken[par] + sh.freed[par];
        const int stop = sh.stop;
        if (stop) {
            if (stop != POOL_LEAVE || nm == 0) break;        // (completed matches first: what is left are frames to enter and parked operands)
            leaving = true;
        }
        par ^= 1u;
    }
    if (sh.stop == POOL_LEAVE && ne) {
        if (tid == 0) { sh.left[0] = ring0; sh.left[1] = avail; sh.left[2] = ne; }
        __syncthreads();
        pool_leave(c, smem, sh);
    }
    if (sh.stop == 2 && tid == 0) c.ctl->pool_exhausted = 1;
    ThreadStats st;
    st.invocations = t.invocations; st.max_depth = t.max_depth;
    st.sc.inserts = t.inserts; st.sc.matches = t.matches;
    flush_stats(c, st);
    pool_report(c, sh.waves, t.max_wave, t.n_late, z.max_calls, z.max_parked, z.fallback, t_start, &sh.next_chunk);
}

// In front of the general scheduler: what the pool kernel could not run (a block ran out of frames: recursion deeper than a
// pool) is seeded again from the start, what blocks have left is put where that scheduler expects it.  False: nothing to do.
__device__ __noinline__ bool pool_take_over(const DevCtx& c, uint32_t& generation) {
    const bool again = c.ctl->pool_exhausted != 0;
    const uint32_t left = c.ctl->hand_mask;
    if (!again && (left == 0u || c.ctl->status != 0)) return false;
    const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = i0; i < c.pool.pair_n; i += stride) reinterpret_cast<uint4*>(c.pair_slots)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (size_t i = i0; i < c.pool.arrived_n; i += stride) c.arrived[i] = 0u;
    for (size_t i = i0; i < c.pool.table_n; i += stride) reinterpret_cast<uint4*>(c.table)[i] = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
    if (again) {
        for (long long b = (long long)i0; b < c.B; b += (long long)stride) seed_instance(c, b);
        if (i0 == 0) {
            Control* k = c.ctl;
            k->invocations = k->tokens = k->store_inserts = k->store_matches = 0ull;
            k->status = 0; k->waves = k->max_wave_tokens = k->max_depth = 0u;
        }
        return grid_barrier(c, &c.ctl->bar.v, generation);
    }
    // frame ids: every call that the pools have made counts as one (those that have come over have the first ones), so that the
    // table is full after as many calls as ever
    if (i0 == 0) c.ctl->frame_count.v = (uint32_t)c.B + (uint32_t)c.ctl->invocations;
    if (!grid_barrier(c, &c.ctl->bar.v, generation)) return false;
    const uint32_t cap = c.pool.cap;
    for (size_t i = i0; i < (size_t)32 * cap; i += stride) {
        const uint32_t slot = (uint32_t)(i / cap), f = (uint32_t)(i % cap);
        if (!((left >> slot) & 1u)) continue;
        const PoolDump d(c, slot);
        const uint32_t id = d.id[f], head = d.head[f];
        if (id == 0xFFFFFFFFu) continue;
        const bool root = head & POOL_ROOT;
        const uint32_t label = root ? 0u : (head >> 16) & 63u;
        uint64_t tag;
        if (c.tag_mode == RDF_TAGS_FRAME) {
            tag = id;
            Frame fr;
            fr.parent = root ? LEAF_MARK : d.id[head & 0xFFFFu]; fr.label = label; fr.arg = d.words[f];
            c.frames[tag] = fr;
            const int n_args = root ? 1 : c.labels[label].n_args;
            for (int k = 1; k < n_args; ++k) c.frame_args[(size_t)tag * 2 + k - 1] = d.words[(size_t)k * cap + f];
        } else {
            uint64_t path = 0;
            uint32_t depth = 0, q = f;
            while (!(d.head[q] & POOL_ROOT) && depth < 64u) {
                path |= (uint64_t)((d.head[q] >> 16) & 63u) << (c.label_bits * depth++);
                q = d.head[q] & 0xFFFFu;
            }
            tag = path_root((long long)(d.head[q] & ~POOL_ROOT)) | (uint64_t)depth << RDF_DEPTH_SHIFT | path;
        }
        if (d.state[f] == 0xFFFFFFFFu) {
            const uint32_t at = atomicAdd(&c.ctl->qcount[0].v, 1u);
            if (at >= c.qcap) {
                set_status(c, RDF_ERR_QUEUE_FULL);
                continue;
            }
            store_token(&c.q[0][at], tag, d.words[f], (uint32_t)(root ? c.result_entry_pc : c.labels[label].entry_pc));
            atomicAdd(&c.ctl->tokens, ~0ull);                // (counted when the call was made, and once more when it is run)
            continue;
        }
        for (int n = 0; n < c.n_match; ++n) {
            const MatchNode M = c.match[n];
            const uint32_t there = d.state[(size_t)n * cap + f] & 0xFFu;
            if (there == (1u << M.n_ports) - 1u) continue;   // (has fired)
            for (int p = 0; p < M.n_ports; ++p) {
                if (!((there >> p) & 1u)) continue;
                const int64_t v = d.words[(size_t)(c.pool.word0 + M.port_base + p) * cap + f];
                StoreCounters sc;                            // (they have been counted)
                int64_t regs[3];
                if (c.tag_mode == RDF_TAGS_FRAME) dense_deliver(c, M, n, tag, p, v, regs, sc);
                else if (hash_insert_or_consume(c, n, tag, v, regs[0], sc) < 0) set_status(c, RDF_ERR_STORE_FULL);
            }
        }
    }
    return grid_barrier(c, &c.ctl->bar.v, generation);
}
