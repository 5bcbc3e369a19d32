// kernels.h -- host launchers of the CUDA kernels in kernels.cu.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "tn_internal.h"

namespace tn {

enum Dtype { DT_I32 = 1, DT_F32 = 2 };

// A batch of B instances sharing one plan: instance b uses the arena slice
// at b * ib bytes and the couplings J + b * jstride, h + b * hstride.
struct Batch {
  int B = 1;
  int64_t ib = 0, jstride = 0, hstride = 0;
};

// Streaming multiprocessors of the current device (queried once per device).
int num_sms();

// Leaves (Sec. II bond / vertex tensors).  x: base of the value arena (bytes),
// counts: when P > 0 every leaf element gets count 1 in each residue plane
// (planes of rbytes = 8- or 4-byte residues).
cudaError_t launch_leaves(Dtype dt, int q, const LeafDesc *d_leaves, int nleaves, const float *J,
                          const float *h, char *arena, int P, int rbytes, const Batch &bt,
                          cudaStream_t st);

// whether every outer index (and a grid stride past it) and every element offset of the
// step fits 32 bits
inline bool gate_fits32(const GateParams &p) {
  int64_t a = 0, b = 0, c = 0, ka = 0, kb = 0, nb = 0, nc = 0;
  for (int s = 0; s < p.nseg; ++s) {
    a += (p.seg_size[s] - 1) * p.seg_sA[s];
    b += (p.seg_size[s] - 1) * p.seg_sB[s];
    c += (p.seg_size[s] - 1) * p.seg_sC[s];
  }
  for (int k = 0; k < p.Ks; ++k) {
    ka = std::max(ka, p.kA[k]);
    kb = std::max(kb, p.kB[k]);
  }
  for (int n = 0; n < p.Ns; ++n) {
    nb = std::max(nb, p.nB[n]);
    nc = std::max(nc, p.nC[n]);
  }
  const int64_t lim = int64_t(1) << 31;
  return p.outer < lim / 2 && a + ka < lim && b + kb + nb < lim && c + nc < lim;
}

// Gate contraction (small B); xA/xB/xC value pointers, nA/nB/nC plane-0
// pointers (counting only).
cudaError_t launch_gate(Dtype dt, const GateParams &p, const void *xA, const void *xB, void *xC,
                        const uint64_t *nA, const uint64_t *nB, uint64_t *nC, const PrimeSet &ps,
                        const Batch &bt, cudaStream_t st);

// Counting gate contraction with compile-time (K, N, planes) forms for 4-byte
// residue planes and for one plane of saturating 64-bit counts (gate_count_*.cu);
// false when the step has no such form (the generic kernel runs it).
bool launch_gate_tc_i32(const GateParams &p, const void *A, const void *B, void *C,
                        const void *nA, const void *nB, void *nC, const PrimeSet &ps,
                        const Batch &bt, cudaStream_t st);
bool launch_gate_tc_f32(const GateParams &p, const void *A, const void *B, void *C,
                        const void *nA, const void *nB, void *nC, const PrimeSet &ps,
                        const Batch &bt, cudaStream_t st);

// Register-tiled max-plus GEMM (128 x 128 tiles, cp.async staging), values only.
// The tile configuration of a shape class is chosen by timing the candidates
// on its first launch outside stream capture (set_gemm_autotune(false) on the
// calling thread skips that and uses the default).
cudaError_t launch_mpgemm(Dtype dt, const GemmParams &p, const void *A, const void *B, void *C,
                          const Batch &bt, cudaStream_t st);
// returns the previous setting of the calling thread
bool set_gemm_autotune(bool on);
// Residue planes of a counting GEMM whose values C were produced already.
cudaError_t launch_gemm_count(Dtype dt, const GemmParams &p, const void *xA, const void *xB,
                              const void *xC, const uint64_t *nA, const uint64_t *nB, uint64_t *nC,
                              const PrimeSet &ps, const Batch &bt, cudaStream_t st);

// Permutation of a tensor (values and, when P > 0, its residue planes).
cudaError_t launch_permute(const PermParams &p, const void *xin, void *xout, const uint64_t *nin,
                           uint64_t *nout, const Batch &bt, cudaStream_t st);

// Argmax traceback over steps [0, nsteps) of d_steps (Sec. III).
// *err is set to 1 if a step meets an unassigned spin (a planning error).
// Records with chain >= 0 refer to d_chains; smem: dynamic shared memory for
// the largest chain record (trace_smem_bytes).
// The spin state (nspins int8) is staged in shared memory during the walk.
cudaError_t launch_trace(Dtype dt, int q, const TraceStep *d_steps, int nsteps,
                         const ChainTrace *d_chains, size_t smem, const char *arena, int8_t *state,
                         int nspins, int *err, const Batch &bt, cudaStream_t st);
size_t trace_smem_bytes(const ChainParams &p, size_t elem);

// The traceback of q = 2 plans whose chains are folded (trace_walk.cu).  A record is a
// list of 32-bit words (encode_walk in program.cpp); tab: element offset of a chain
// record's gate tables in the instance's arena slice (ntab values).
constexpr int kWalkTable = TN_CHAIN_MAX_G * TN_TG_TABLE;
constexpr int kWalkRec = 8 + 7 * TN_MAX_TRACE_LEGS;
struct WalkIdx {
  int64_t tab;
  int32_t rec, len, ntab, pad;
};
struct WalkArgs {
  const int32_t *recs = nullptr;       // device: record words
  const WalkIdx *idx = nullptr;        // device: this trace's records
  int n = 0;
  const int32_t *list = nullptr;       // device: (record, chain) of its chain records
  int nlist = 0;
  const ChainTrace *chains = nullptr;  // device
  int64_t best = -1;                   // arena byte offset of the wide search's key
  // records searched by a grid, in order: position, record word, contracted states
  int nbig = 0;
  const int *big = nullptr, *big_rec = nullptr;
  const int64_t *big_k = nullptr;
};
cudaError_t launch_walk(Dtype dt, const WalkArgs &w, char *arena, int8_t *state, int nspins,
                        int *err, const Batch &bt, cudaStream_t st);

// Tables of best completions along a frontier plan (device copies of its records) and S
// samples drawn from them (sample_frontier.cu): X, N of p.elements entries, sigma S x n.
// *err (device) is set to 1 when a draw fails; *launches grows by the kernels launched.
struct FrontierPlan;
struct FrontierStep;
struct FrontierNb;
cudaError_t launch_frontier_sample(const FrontierPlan &p, const FrontierStep *steps,
                                   const FrontierNb *nbs, int32_t *X, uint64_t *N, int S,
                                   uint64_t seed, int8_t *sigma, int *err, int *launches,
                                   cudaStream_t st);

// A run of small steps in one launch, one block per instance.  Descriptors (32-bit
// words): {steps, levels}, level starts [levels + 1], outputs of each level, per step its
// first output within its level, per step the word of its body, then the bodies: 64-bit
// offsets of the values of A, B (-1: none) and C (-1: not stored) in elements and of their
// counts in 8-byte words, digits, K, N, flags (1: B counts 1; 2, 4: the rule for NaN),
// shared-memory elements of A, B and C
// (-1: not there), then (size, stride in A, stride in B) of each outer digit (slowest
// first), (offset in A, in B) of each k, the offset in B of each n (N > 1).  words is a
// multiple of 4; scratch: shared-memory elements.  sat: one plane of saturating 64-bit
// counts.
constexpr int kSmallMaxWords = 40 * 1024;     // descriptor words of a run at most
constexpr int kSmallScratch = 5 * 1024;       // shared-memory elements at most (12 bytes each)
cudaError_t launch_small(Dtype dt, bool sat, const int32_t *d_desc, int words, int scratch,
                         char *arena, const Batch &bt, cudaStream_t st);

// Fused gate chain over tiles of the big tensor (values; planes when P > 0).
cudaError_t launch_chain(Dtype dt, const ChainParams &p, const char *arena, const void *Ax,
                         const uint64_t *An, void *Cx, uint64_t *Cn, const PrimeSet &ps,
                         const Batch &bt, cudaStream_t st);
size_t chain_smem_bytes(const ChainParams &p, size_t elem);

// Folded register chain of INT32 values with one plane of saturating 64-bit
// counts (chain_sat.cu).
cudaError_t launch_schain(const ChainParams &p, const char *arena, const void *Ax,
                          const uint64_t *An, void *Cx, uint64_t *Cn, const Batch &bt,
                          cudaStream_t st);

// Sum of n = 2 or 4 gate contractions over the same output indices (gate_sum.cu):
// n = 2: G0 + G1, n = 4: (G0 + G1) + (G2 + G3); counts multiply (the forms it takes:
// gate_sum_leaf in program.cpp).
constexpr int TN_SUM_MAX_G = 4;
struct GateSum {
  int32_t n = 0, nseg = 0, Ns = 0;
  int64_t outer = 0;
  int32_t seg_size[TN_MAX_SEG], seg_sh[TN_MAX_SEG], seg_sC[TN_MAX_SEG];
  int32_t seg_sA[TN_SUM_MAX_G][TN_MAX_SEG];
  int32_t kA[TN_SUM_MAX_G][2], kB[TN_SUM_MAX_G][2], nB[TN_SUM_MAX_G][TN_GATE_MAX_N];
};
cudaError_t launch_gate_sum(Dtype dt, bool cnt, const GateSum &p, const void *const *A,
                            const void *const *B, const uint64_t *const *nA, void *C,
                            uint64_t *nC, const Batch &bt, cudaStream_t st);

// Fused gate chain of q = 3 values (chain3.cu).
cudaError_t launch_chain3(Dtype dt, const ChainParams &p, const char *arena, const void *A,
                          void *C, const Batch &bt, cudaStream_t st);

// Resident blocks of a kernel on the whole device and the grid (blocks per
// instance) of a grid-stride kernel with `need` blocks of work per instance.
int64_t wave_blocks(int64_t need, int B, int64_t slots);

// dE/dJ and dE/dh at the traced state.
cudaError_t launch_grad(int q, int n, int m, const int32_t *eu, const int32_t *ev,
                        const int8_t *state, float *dJ, float *dh, int B, cudaStream_t st);

// Convert a state (indices) to the +-1 / 0..q-1 convention of tn_config.
cudaError_t launch_state_out(int q, int n, const int8_t *state, int8_t *out, int B,
                             cudaStream_t st);

// Static scratch of tn_energy_noalloc (noalloc.cu): its size, its device
// address on the current device (looked up once per device), and the kernel
// writing E = -root as float.
size_t noalloc_scratch_bytes();
cudaError_t noalloc_scratch(char **ptr);
cudaError_t launch_energy_out(Dtype dt, const void *root, float *E, cudaStream_t st);
// Leaves of tn_energy_noalloc from host descriptors passed as kernel
// parameters (no device copy of the descriptors; values only).
cudaError_t launch_leaves_param(Dtype dt, int q, const LeafDesc *leaves, int nleaves,
                                const float *J, const float *h, char *scratch, cudaStream_t st);

}  // namespace tn
