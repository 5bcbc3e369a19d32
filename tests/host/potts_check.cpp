// potts_check.cpp -- host check of the programs of Potts (q = 3) plans (no GPU).  The
// program without small runs (the allocation-free energy's) has the chains of the one with
// them, on tiles of eight legs where the state has that many; orders are scored with tiles of
// seven, whose arena is within 1 KB of it.  Prints "programs N wide W bad 0".
#include <cstdio>
#include <string>
#include "program.h"
namespace tn {
size_t trace_smem_bytes(const ChainParams &p, size_t elem) { return elem * (size_t)(p.ngates + 1) * p.tile; }
size_t chain_smem_bytes(const ChainParams &, size_t) { return 0; }
}
using namespace tn;
static Net potts(int L, int W) {
  Net n; n.n = L * W; n.q = 3;
  for (int i = 0; i < L; ++i) for (int j = 0; j < W; ++j) { int s = i * W + j;
    if (j + 1 < W) { n.eu.push_back(s); n.ev.push_back(s + 1); }
    if (i + 1 < L) { n.eu.push_back(s); n.ev.push_back(s + W); } }
  n.m = (int)n.eu.size(); for (int e = 0; e < n.m; ++e) n.J.push_back(1.f);
  n.build_leaves(); return n;
}
int main() {
  int programs = 0, wide = 0, bad = 0;
  for (int L : {9, 11, 13}) for (int W : {8, 10, 11, 12, 13}) for (int greedy : {0, 1}) {
    Net net = potts(L, W);
    Tree t; std::string err;
    if (!greedy) { std::vector<int> seq(net.n); for (int i = 0; i < net.n; ++i) seq[i] = i; if (!tree_from_sweep(net, seq, &t, &err)) return 2; }
    else { CostModel cm; if (!tree_greedy(net, 5 + W, 4, cm, &t, &err)) return 2; }
    Plan pl; if (!classify(net, t, &pl, &err)) return 2;
    Program run, flat, score;
    if (!build_program(net, pl, PM_ENERGY, DT_F32, 0, 0, &run, &err)) return 2;
    if (!build_program(net, pl, PM_ENERGY, DT_F32, 0, 0, &flat, &err, 8, false, false)) return 2;
    if (!build_program(net, pl, PM_ENERGY, DT_F32, 0, 0, &score, &err, 8, false, false, true)) return 2;
    programs++;
    bool same = run.chains.size() == flat.chains.size();
    for (size_t i = 0; same && i < run.chains.size(); ++i) {
      same = run.chains[i].t == flat.chains[i].t && run.chains[i].ngates == flat.chains[i].ngates &&
             run.chains[i].outer == flat.chains[i].outer;
      wide += flat.chains[i].t == 8;
    }
    for (const ChainParams &p : score.chains) same = same && p.t <= 7;
    if (!same || flat.arena_bytes > score.arena_bytes + 1024) {
      std::printf("L %d W %d greedy %d: chains %zu %zu arena %lld %lld\n", L, W, greedy, run.chains.size(), flat.chains.size(),
                  (long long)flat.arena_bytes, (long long)score.arena_bytes);
      bad++;
    }
  }
  std::printf("programs %d wide %d bad %d\n", programs, wide, bad);
  return bad != 0;
}
