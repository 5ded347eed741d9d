// The candidates of pd_autotune and its cache lines, "key|block split pairs ring automatic".  No CUDA here: a host
// test compiles it.
#pragma once

#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

namespace pd {

// A launch mapping: the options it stands for, or the automatic shapes (with the resident kernels where they apply).
struct TuneChoice {
  int block = -1, split = -1, pairs = -1, ring = -1;
  bool automatic = false;
};

// The mappings that are timed.  The automatic one comes first wherever it is more than one (block, split): the FP64
// forms give pass 1a a shape of its own and small bodies the resident kernel, and the lattice kernels a ring beside
// their block, so that no explicit mapping stands for what an untuned context runs.
inline std::vector<TuneChoice> tune_candidates(bool fp64, bool lattice, bool try_pairs, int pairs, int ring) {
  std::vector<TuneChoice> r;
  const int npairs = try_pairs ? 2 : 1;
  auto add = [&](int block, int split, int k, int rg, bool automatic) {
    TuneChoice t;
    t.block = block;
    t.split = split;
    t.pairs = try_pairs ? 1 - k : pairs;
    t.ring = rg;
    t.automatic = automatic;
    r.push_back(t);
  };
  if (fp64 || lattice)
    for (int k = 0; k < npairs; ++k) add(256, 1, k, ring, true);  // (the options as a new context has them)
  for (int block : {64, 128, 256, 512})
    for (int split : {1, 2, 4}) {
      if ((block / 32) % split) continue;
      if (lattice && split != 1) continue;  // the lattice kernels run one warp per slice
      for (int k = 0; k < (lattice ? 4 : npairs); ++k) add(block, split, lattice ? 0 : k, lattice ? k : ring, false);
    }
  return r;
}

// What the fastest mapping depends on.  Everything that decides which kernels a step runs belongs to it: a choice
// made for one form (nonlinear bonds, say, which have no resident kernel in FP64) must not be taken for another.
struct TuneProblem {
  long long n = 0, bonds = 0, entries = 0;
  int dim = 0, precision = 0, bodies = 0, kinematics = 0, solver = 0, influence = 0;
  int lattice = 0, shadow_lo = 0, bond_cache = 0, stage = 0, validate = 0, resident = 0;
  std::string device;
};

inline std::string tune_key(const TuneProblem& p) {
  char s[384];
  std::snprintf(s, sizeof(s),
                "osbpd-2 n=%lld bonds=%lld entries=%lld dim=%d prec=%d bodies=%d kin=%d solver=%d infl=%d lattice=%d lo=%d "
                "cache=%d stage=%d validate=%d resident=%d dev=",
                p.n, p.bonds, p.entries, p.dim, p.precision, p.bodies, p.kinematics, p.solver, p.influence, p.lattice,
                p.shadow_lo, p.bond_cache, p.stage, p.validate, p.resident);
  std::string key = std::string(s) + p.device;
  for (char& c : key)
    if (c == '\n' || c == '|') c = ' ';
  return key;
}

inline std::string tune_line(const std::string& key, const TuneChoice& t) {
  char s[96];
  std::snprintf(s, sizeof(s), "|%d %d %d %d %d\n", t.block, t.split, t.pairs, t.ring, t.automatic ? 1 : 0);
  return key + s;
}

// True when the line is this key's: all five numbers, or it says nothing about the automatic mapping.
inline bool tune_parse(const char* line, const std::string& key, TuneChoice* t) {
  const char* bar = std::strchr(line, '|');
  if (!bar || std::string(line, bar) != key) return false;
  TuneChoice r;
  int am = 0;
  if (std::sscanf(bar + 1, "%d %d %d %d %d", &r.block, &r.split, &r.pairs, &r.ring, &am) != 5) return false;
  r.automatic = am != 0;
  *t = r;
  return true;
}

}  // namespace pd
