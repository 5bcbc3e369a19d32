// program.h -- lowering of a classified contraction plan to a fixed sequence
// of kernel launches with statically planned arena offsets.
#pragma once
#include <cstdint>
#include <string>
#include <vector>

#include "kernels.h"
#include "planner.h"
#include "tn_internal.h"

namespace tn {

// Location of a tensor: byte offsets inside a buffer (values at xoff, residue
// plane 0 at noff, planes `plane` elements apart).
struct Loc {
  int buf = -1;
  int64_t xoff = 0, noff = 0, plane = 0;
};

struct BufInfo {
  int64_t bytes = 0;
  int first = 1 << 30, last = -1;
  int64_t off = -1;
};

enum OpKind { OP_LEAVES, OP_PERM, OP_GATE, OP_GEMM, OP_TRACE, OP_CHAIN, OP_SMALL, OP_GSUM };

struct Op {
  OpKind kind;
  Loc in0, in1, out;
  int idx = -1;              // into gates / gemms / perms
  int trace_begin = 0, trace_n = 0;
  double bytes = 0, macs = 0;  // algorithmic traffic and multiply-adds of the launch
};

// A run of small steps (gates, transposes, GEMMs of few elements) that one block per
// instance executes in one launch: ops sorted by dependency level, level l being
// ops [level[l], level[l + 1]).  The encoded descriptors (kernels.h) start at int
// desc_off of the program's descriptor array.
struct SmallRun {
  std::vector<Op> ops;
  std::vector<int> level;
  int64_t desc_off = 0;
  int desc_len = 0, scratch = 0;       // descriptor words, shared-memory elements
};

// A product of gate contractions (gate_sum.cu) and its operands.
struct SumOp {
  GateSum p;
  std::vector<Loc> A, B;
};

// One traceback launch of a q = 2 plan with folded chains: records [begin, begin + n)
// of the trace, the buffer of its chains' gate tables and of the wide searches' key.
struct Walk {
  int begin = 0, n = 0;
  Loc tables, best;
  std::vector<int64_t> toff;           // per record: its tables' first element
  int idx_off = 0, list_off = 0, nlist = 0;
  std::vector<int> big, big_rec;       // see WalkArgs
  std::vector<int64_t> big_k;
};

enum ProgMode { PM_ENERGY = 0, PM_CONFIG = 1, PM_COUNT = 2 };

struct Program {
  ProgMode mode;
  Dtype dt;
  int q = 2, P = 0;
  int rbytes = 8;                    // bytes of one residue of the counting planes
  bool pass_prime = false;           // one 31-bit prime per pass: plane 0's prime is set per run
  bool sat = false;                  // one 8-byte plane of exact, saturating 64-bit counts
  std::vector<BufInfo> bufs;
  std::vector<Op> ops;
  std::vector<GateParams> gates;
  std::vector<GemmParams> gemms;
  std::vector<PermParams> perms;
  std::vector<SmallRun> smalls;
  std::vector<SumOp> gsums;
  std::vector<int32_t> small_desc;                  // descriptors of every run
  std::vector<ChainParams> chains;                  // fused gate chains
  std::vector<const void *> chain_jit;              // their compiled kernels (nullptr: interpreted)
  std::vector<std::vector<Loc>> chain_blocs;        // their gate operands
  std::vector<ChainTrace> chain_traces;             // traceback records of chains
  std::vector<Loc> ctrace_in;
  std::vector<Walk> walks;                          // of OP_TRACE ops with idx >= 0
  std::vector<int32_t> walk_words, walk_list;
  std::vector<WalkIdx> walk_idx;
  std::vector<std::vector<Loc>> ctrace_blocs;
  size_t trace_smem = 0;                            // dynamic smem of the trace kernel
  std::vector<LeafDesc> leaves;      // offsets absolute after planning
  std::vector<TraceStep> trace;      // offsets absolute after planning
  std::vector<Loc> traceA, traceB;
  Loc leaves_loc;
  std::vector<int64_t> leaf_elem;    // element offset of each leaf in the leaves buffer
  Loc root;
  int64_t arena_bytes = 0;
  int fwd_end = 0;                   // ops [0, fwd_end) are the forward pass
  int n_transposes = 0, n_gate = 0, n_gemm = 0, n_recompute = 0, n_chain = 0, n_chain_gates = 0;
  double macs = 0;                   // tropical multiply-adds of the forward steps
  // CUDA graphs of op ranges, captured on the second run of a range
  struct Graph {
    int begin, end, runs, B;
    const char *arena;
    const float *J, *h;
    const int8_t *state;
    cudaGraphExec_t exec;
  };
  std::vector<Graph> graphs;
  // device copies (owned by the context)
  LeafDesc *d_leaves = nullptr;
  int32_t *d_small = nullptr, *d_walk = nullptr, *d_walk_list = nullptr;
  WalkIdx *d_walk_idx = nullptr;
  TraceStep *d_trace = nullptr;
  ChainTrace *d_chain_traces = nullptr;
};

// Build the program for a plan.  seg_bytes: traceback checkpoint segment
// budget (PM_CONFIG; <= 0 keeps every intermediate).
// rbytes: bytes of one residue of the counting planes (8: 61-bit primes; 4:
// 31-bit primes, the one-prime-per-pass counts).  sat (PM_COUNT, P = 1, rbytes
// = 8): the plane holds exact, saturating counts.  small_runs: group the small
// steps of the forward pass into runs (value and exact-count programs).  scoring: the
// program is not run but ranks an order in the search (no runs either).
bool build_program(const Net &net, const Plan &plan, ProgMode mode, Dtype dt, int P,
                   int64_t seg_bytes, Program *pr, std::string *err, int rbytes = 8,
                   bool sat = false, bool small_runs = true, bool scoring = false);

int64_t abs_off(const Program &pr, const Loc &l);  // arena byte offset of values

}  // namespace tn
