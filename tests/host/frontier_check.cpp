// Host check of the frontier plans behind tn_sample: the tables of a plan, evaluated
// here, must give the draws of the prefix-by-prefix sampler (sampler.cpp) with
// brute-force counts, for any order, with and without fields, isolated spins and ties.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "sampler.h"

using namespace tn;

int main() {
  std::mt19937 rng(7);
  int bad = 0, wide = 0;
  for (int it = 0; it < 120; ++it) {
    const int n = 1 + (int)(rng() % 9);
    std::vector<int> eu, ev, order(n);
    std::vector<float> J, h(n, 0.f);
    for (int i = 0; i < n; ++i)
      for (int j = i + 1; j < n; ++j)
        if (rng() % 3 == 0) {
          eu.push_back(rng() % 2 ? i : j);
          ev.push_back(eu.back() == i ? j : i);
          J.push_back((float)((int)(rng() % 5) - 2));
        }
    if (it % 2) for (float &x : h) x = (float)((int)(rng() % 3) - 1);
    for (int i = 0; i < n; ++i) order[i] = i;
    if (it % 3) std::shuffle(order.begin(), order.end(), rng);
    CountFn brute = [&](const std::vector<float> &hh, int K, std::vector<double> *E,
                        std::vector<Big> *cnt) {
      E->assign(K, 0);
      cnt->assign(K, Big());
      for (int k = 0; k < K; ++k) {
        double best = INFINITY;
        uint64_t c = 0;
        for (unsigned x = 0; x < (1u << n); ++x) {
          auto s = [&](int i) { return (x >> i & 1) ? -1.0 : 1.0; };
          double e = 0;
          for (size_t m = 0; m < eu.size(); ++m) e -= J[m] * s(eu[m]) * s(ev[m]);
          for (int i = 0; i < n; ++i) e -= hh[(size_t)k * n + i] * s(i);
          if (e < best) { best = e; c = 1; } else if (e == best) ++c;
        }
        (*E)[k] = best;
        (*cnt)[k] = Big{c};
      }
      return 0;
    };
    const int S = 5;
    const uint64_t seed = rng();
    std::vector<int8_t> want, got((size_t)S * n);
    std::string err;
    if (sample_ground_states(n, S, order, h, seed, 16, brute, &want, &err)) ++bad;
    FrontierPlan fp;
    if (!plan_frontier(n, eu, ev, J, h, order, 26, &fp)) { ++bad; continue; }
    std::vector<int> X(fp.elements, 0);
    std::vector<uint64_t> N(fp.elements, 1);
    auto field = [&](const FrontierStep &st, uint32_t i) {
      int z = st.h;
      for (int k = st.nb; k < st.nb + st.nnb; ++k)
        z += (i >> fp.nbs[k].slot) & 1 ? -fp.nbs[k].J : fp.nbs[k].J;
      return z;
    };
    for (int t = n - 1; t >= 0; --t) {
      const FrontierStep &st = fp.steps[t];
      if (t + 1 < n && st.next != fp.steps[t + 1].off) ++bad;
      for (uint32_t i = 0; i < st.size; ++i) {
        const uint32_t up = i & st.keep, dn = st.slot >= 0 ? up | (1u << st.slot) : up;
        const uint32_t behind = t + 1 < n ? fp.steps[t + 1].size : 1;
        if (up >= behind || dn >= behind) { ++bad; continue; }
        const int z = field(st, i), a = X[st.next + up] + z, b = X[st.next + dn] - z;
        X[st.off + i] = std::max(a, b);
        N[st.off + i] = (a >= b ? N[st.next + up] : 0) + (b >= a ? N[st.next + dn] : 0);
      }
    }
    for (int s = 0; s < S; ++s) {
      uint32_t state = 0;
      for (int t = 0; t < n; ++t) {
        const FrontierStep &st = fp.steps[t];
        if (state >= st.size) { ++bad; break; }
        const uint32_t up = state & st.keep, dn = st.slot >= 0 ? up | (1u << st.slot) : up;
        const int z = field(st, state), a = X[st.next + up] + z, b = X[st.next + dn] - z;
        const uint64_t wp = a >= b ? N[st.next + up] : 0, wm = b >= a ? N[st.next + dn] : 0;
        const bool plus = big_less(uniform_below(Big{wp + wm}, seed, s, t), Big{wp});
        got[(size_t)s * n + st.spin] = plus ? 1 : -1;
        state = plus ? up : dn;
      }
    }
    if (got != want) ++bad;
    // a frontier wider than allowed is refused
    int w = 0;
    for (const auto &st : fp.steps) w = std::max(w, st.slot + 1);
    if (w > 0 && plan_frontier(n, eu, ev, J, h, order, w - 1, &fp)) ++bad;
    wide = std::max(wide, w);
  }
  std::printf("widest %d bad %d\n", wide, bad);
  return bad != 0 || wide < 4;
}
