// sampler.h -- uniform sampling of ground states by conditional counts.
//
// Sec. III: besides backtracking, ground states can be drawn by fixing the
// spins one at a time in an arbitrary order, each with its conditional
// probability of being in a ground state given the spins fixed before it.
// With exact degeneracy counts this gives every ground state the same
// probability 1/count.
//
// Conditioning uses fields.  Add a field p_j in {+1, -1} to every fixed spin
// j (k of them).  A state agreeing with all k pins has E' = E - k; one that
// disagrees on at least one has E' >= E - (k - 2).  So the pinned instance
// has minimum E_min - k exactly when some ground state agrees with the pins,
// and then its minimisers are exactly those ground states: its count is the
// number of ground states with that prefix.  (Any positive pin strength
// works; 1 keeps integral instances integral and exact.)
//
// This file is host logic only: the counts come from a callback (the library
// passes batched GPU contractions, the host tests pass brute force).
#pragma once
#include <cstdint>
#include <functional>
#include <string>
#include <vector>

namespace tn {

// Unsigned big integer, little-endian 64-bit limbs (no leading-zero limbs
// required).
typedef std::vector<uint64_t> Big;

// Counts K pinned instances.  h holds K field vectors of n floats each; on
// success E[k] is the minimum energy and cnt[k] the number of minimisers of
// instance k.  Returns 0, or a nonzero status that the sampler passes on.
typedef std::function<int(const std::vector<float> &h, int K, std::vector<double> *E,
                          std::vector<Big> *cnt)>
    CountFn;

// Draw S ground states of an Ising instance with n spins and fields h0
// (zeros when it has none), fixing spins in `order` (a permutation of
// 0..n-1).  At most `chunk` samples share one batch of 2 * chunk counts.
// sigma: S * n values +-1, sample-major.  Sample s draws its random numbers
// from a counter-based generator keyed by (seed, s, step), so a sample does
// not depend on S or chunk.  Returns 0 or the callback's status; *err says
// why (a status of -1 means the counts were inconsistent).
int sample_ground_states(int n, int S, const std::vector<int> &order, const std::vector<float> &h0,
                         uint64_t seed, int chunk, const CountFn &count,
                         std::vector<int8_t> *sigma, std::string *err);

// The spins of an order as a sweep of one frontier.  Behind step t stand the placed spins
// that still have a neighbour to come; spin order[t] takes a slot (one bit of a state
// index) unless none of its neighbours comes later, and a spin whose last neighbour is
// placed gives its slot back before the new one is taken.
struct FrontierStep {
  int64_t off;            // first element of the table in front of this step
  int64_t next;           // first element of the table behind it
  uint32_t size;          // states of the table (bits of free slots make no difference)
  uint32_t keep;          // slots that stay
  int32_t slot, spin;     // slot of the new spin (-1: none) and its number
  int32_t h;              // its field
  int32_t nb, nnb;        // its earlier neighbours: [nb, nb + nnb) of the array below
  int32_t pad;
};
struct FrontierNb {
  int32_t slot, J;
};
struct FrontierPlan {
  std::vector<FrontierStep> steps;
  std::vector<FrontierNb> nbs;
  int64_t elements = 0;   // of all tables, the one behind the last step included
};
// false: a frontier of more than max_bits slots (couplings J, h must be integral)
bool plan_frontier(int n, const std::vector<int> &eu, const std::vector<int> &ev,
                   const std::vector<float> &J, const std::vector<float> &h,
                   const std::vector<int> &order, int max_bits, FrontierPlan *out);

// Helpers (exposed for tests).
uint64_t mix64(uint64_t x);                         // SplitMix64 finaliser
bool big_less(const Big &a, const Big &b);
Big big_add(const Big &a, const Big &b);
Big uniform_below(const Big &bound, uint64_t seed, uint64_t s, uint64_t step);

}  // namespace tn
