// Internal structures shared by the host-side graph builder and the device
// executor.  Not part of the public boundary (see include/rdf.h).
#pragma once
#include <stdint.h>

#include <string>
#include <vector>

#include "rdf.h"

// ---------------------------------------------------------------------------
// Lowered device program.
//
// The static graph is cut into *segments*: maximal pieces that one arriving
// token (or one completed match) can run through without waiting for another
// token.  A segment is straight-line/branching code for a small register
// machine; the tag operations and the token-store accesses are instructions.
// ---------------------------------------------------------------------------
enum VmOp : uint8_t {
    VM_MOVI = 0,   // r[dst] = imm
    VM_MOVC,       // r[dst] = const_pool[imm]
    VM_MOV,        // r[dst] = r[a]
    VM_ADD, VM_SUB, VM_MUL, VM_MAX, VM_LT, VM_EQ, VM_REM,   // r[dst] = r[a] op r[b]
    VM_ISLEAF, VM_LEFT, VM_RIGHT, VM_TOK,           // r[dst] = tree accessor(r[a])
    VM_BRZ,        // Switch: if r[a] == 0 jump to imm (segment-relative before layout, absolute after)
    VM_JMP,        // jump to imm
    VM_CALL,       // Call_i: push label imm on the tag, send <i:t, r[a]> (further parameters r[b], r[dst]) to the callee
    VM_CALL_A,     // a Call_i that is followed in straight-line code by another one (VM_CALL_B): reserves frames and queue
    VM_CALL_B,     //   slots for both at once (one round of atomics on the token's critical path instead of two)
    VM_LDARG,      // r[dst] = parameter imm (> 0) of this invocation, kept in its frame
    VM_PORT,       // deliver r[a] to input port b of match node imm under the current tag
    VM_RET,        // the function's output r[a]: Return_i pops the tag and continues in the caller
    VM_OUT,        // r[a] is the program's output for this instance
    VM_EMBED,      // leaf state: queue E[r[a]] -> state of this frame; continue at segment imm next wave
    VM_LEAF_LSTM,  // same for the TreeLSTM leaf
    VM_ENTER,      // Enter: new loop frame under the current tag, counter 0; variables r[a], r[b], r[dst]; loop head at imm
    VM_NEXT,       // Next: counter + 1, variables r[a], r[b], r[dst], back to the loop head at imm (next wave)
    VM_EXIT,       // Exit: the tag below the loop frame again; carries on in the same segment
    VM_VCHILD,     // unary vector operator dst (0 left, 1 right half of W) on the state r[a] -> state of this frame; continue at imm next wave
    VM_VGATE,      // r[dst] = W_s[0] . state(r[a]) + b_s[0] > 0: an integer read off a vector value
    VM_HALT
};

struct VmInstr {
    uint8_t op, dst, a, b;
    int32_t imm;
};

enum MatchKind : int32_t { MATCH_INT = 0, MATCH_CELL_RNN = 1, MATCH_CELL_LSTM = 2 };

struct MatchNode {
    int32_t n_ports;     // tagged inputs that must meet
    int32_t kind;        // MatchKind
    int32_t cont_pc;     // INT: code run with r0..r(n-1) = port values; CELL_*: code run next wave with r0 = state slot
    int32_t port_base;   // first port in the dense (frame-mode) port array
};

enum ContKind : int32_t { K_PORT = 0, K_SEG = 1, K_RET = 2 };

struct LabelInfo {
    int32_t entry_pc;    // entry segment of the callee
    int32_t k_kind;      // what Return_i feeds: ContKind
    int32_t k_node;      // K_PORT: match node
    int32_t k_port;      // K_PORT: its port
    int32_t k_pc;        // K_SEG: code run with r0 = returned value
    int32_t child_index; // position of this call site among the call sites of its caller's body
    int32_t callee;      // function index
    int32_t local_label; // i of Call_i in the per-callee numbering of Section 3
    int32_t n_args;      // formal parameters of the callee (one Call_i node per parameter)
};

static const int RDF_MAX_REGS = 16;
static const int RDF_MAX_LABELS = 64;
static const int RDF_MAX_MATCH = 16;
static const int RDF_MAX_CODE = 1024;
static const int RDF_MAX_CONSTS = 64;
static const int RDF_PATH_BITS = 38;       // packed path field
static const int RDF_DEPTH_SHIFT = 38;     // 6-bit depth field above it
static const int RDF_INST_SHIFT = 44;      // 20-bit instance field

// ---------------------------------------------------------------------------
// The lowered program of an integer graph once more, fused for the pool executor
// (rdf_pool.cuh): operands are register + immediate, a comparison branches by
// itself.  Small programs only; the kernel gets it as a parameter.
// ---------------------------------------------------------------------------
enum PoolOp : uint8_t {
    PI_HALT = 0, PI_BR, PI_RET, PI_CALL, PI_PORT, PI_ADD, PI_SUB, PI_MUL, PI_MAX, PI_REM, PI_CMP, PI_MOV, PI_CONST, PI_ARG, PI_JMP,
    PI_TREE, PI_OUT
};
enum PoolCmp : uint8_t { PC_LT = 0, PC_EQ, PC_NE };
enum PoolTree : uint8_t { PT_ISLEAF = 0, PT_LEFT, PT_RIGHT, PT_TOK };

struct alignas(16) PoolInstr {
    uint8_t op, dst, cmp, n_run;     // cmp: PoolCmp / PoolTree / port; n_run: calls that follow one another from here
    uint8_t ra, rb, rc;              // operand registers (n_regs: the zero register) ...
    uint8_t last : 1, tail : 1;      // nothing follows in the segment; the call is the caller's own output
    int32_t ia, ib, ic;              // ... plus immediates
    int32_t imm;                     // branch target, label, match node, constant, parameter
    int32_t pad[2];
};
struct alignas(16) PoolLabel {
    int16_t entry, k_pc;
    uint8_t k_kind, k_node, k_port, n_args;
    int32_t fast;                    // PoolProgram::entry_of its callee, -1: run by the interpreter
    int32_t pad;
};
struct PoolMatch {
    int16_t  cont;
    uint8_t  n_ports, word0;         // its ports are words word0 .. of the frame
    uint32_t all;                    // a bit per port
};
// Common shapes of a segment, run without the interpreter, everything in registers (operand registers 0 .. 2: the arguments
// or the operands of the match; 3: zero).
struct PoolOperand { int32_t reg, imm; };
struct alignas(16) PoolAction {                  // return ops[0], or make n_calls calls with 3 operands each
    int32_t n_calls, labels[3];                  // n_calls 0: return; label | arguments << 8
    PoolOperand ops[9];
    int32_t pad[2];
};
struct alignas(16) PoolEntry {                   // entering a function: the action of the first condition that holds, else the last one
    int32_t n_cond, n_args, cmp[2];              // n_cond -1: not of this shape
    PoolOperand a[2], b[2];
    PoolAction act[3];
};
struct alignas(16) PoolCont {                    // after a match: return `a op b` + imm, or (op PI_CALL) the caller's own output is a call
    int32_t op, imm;                             // op PI_HALT: not of this shape
    PoolOperand a, b;
    PoolOperand ops[3];
    int32_t label;
    int32_t pad[3];
};
static const int POOL_MAX_ENTRY = 4, POOL_MAX_CONT = 2;
static const int POOL_MAX_CODE = 48, POOL_MAX_LABELS = 16, POOL_MAX_MATCH = 8, POOL_MAX_CONSTS = 4, POOL_MAX_WORDS = 8;
struct alignas(16) PoolProgram {
    int32_t   n_code, n_labels, n_match, result_entry;
    int32_t   words, n_regs;         // 64-bit words per frame, registers per thread
    int32_t   calls_entry, calls_cont;   // most frames taken by a segment that enters a function / that carries on after a match
    int32_t   late_calls, tails, word0, pad;   // some call waits for another one; some call takes over its caller's frame; word of port 0
    PoolInstr code[POOL_MAX_CODE];
    PoolLabel labels[POOL_MAX_LABELS];
    PoolMatch match[POOL_MAX_MATCH];
    int64_t   consts[POOL_MAX_CONSTS];
    PoolEntry entry_of[POOL_MAX_ENTRY];
    PoolCont  cont_of[POOL_MAX_CONT];    // by match node
};

// A program of one recursive function whose body returns a value or makes n_ports calls that meet in one operator (rdf_lanes.cuh).
// Operands of conditions, returned values and calls: over the parameters; of the operator: over its operands in the order the calls
// are made; of `root`: over the program's argument.
struct LaneOperand { uint64_t mask[3]; int64_t imm; };      // the value whose mask is set, plus a constant
struct LaneProgram {
    int32_t n_args, n_ports;
    int32_t n_cond, call_at, cmp[2];             // the first condition that holds: its action, else the last one; call_at: the one that makes the calls
    int32_t cont, ret_at;                        // PI_ADD .. PI_MAX: ca op cb + cont_imm is returned; PI_CALL: `tail` are the parameters of the same function
    int64_t cont_imm, out_imm;
    LaneOperand a[2], b[2];
    LaneOperand ret[2];                          // returned by the other actions, the second one by action ret_at
    LaneOperand call[9], root[3];                // parameters of the calls, 3 each; of the call `result` makes
    LaneOperand ca, cb, tail[3];
    int32_t label[4], port[3];                   // labels of the calls, and (3) of the one `result` makes; the operator's ports they feed
};

struct rdf_graph {
    // literal graph (Section 3 transformation), for inspection
    std::vector<rdf_node> nodes;
    std::vector<rdf_edge> edges;
    // lowered program
    std::vector<VmInstr> code;
    std::vector<MatchNode> match;
    std::vector<LabelInfo> labels;
    std::vector<int64_t> consts;
    std::vector<int32_t> label_callee, label_local;   // the same two fields of `labels`, as plain arrays for rdf_graph_describe
    std::vector<int32_t> label_caller;                // per label: the function whose body makes the call
    int32_t result_entry_pc = 0;
    int32_t n_ports_total = 0;
    int32_t max_calls_per_body = 1;
    int32_t max_params = 1;
    int32_t label_bits = 1;
    int32_t tag_mode = RDF_TAGS_PATH;
    bool has_vector_ops = false;
    bool has_rnn = false, has_lstm = false, has_loss = false;
    bool uses_tree = false;
    bool has_loops = false;
    // structural recursion over the input trees (rdf_fold.cuh): f(v) = leaf(tok v) or cell(f(child), f(child)), result(v) = f(v)
    bool fold = false;
    int32_t fold_label[3] = {0, 0, 0};    // label ids of the calls of operand 0 and operand 1 and of `result`'s call
    int32_t fold_right[2] = {0, 1};       // the child that operand 0 / 1 descends into: 0 left, 1 right
    bool pool = false;            // an integer program that fits the pool executor
    PoolProgram pool_prog{};
    bool lanes = false;           // a call per thread
    LaneProgram lane_prog{};
    bool interleaved = false;     // some Switch reads a vector value: operators run between the token waves
    std::vector<std::string> func_names;
    // per-run state owned by the executor (rdf_exec.cu)
    void* dev = nullptr;
};

// implemented in rdf_exec.cu
void rdf_exec_release(rdf_graph* g);
