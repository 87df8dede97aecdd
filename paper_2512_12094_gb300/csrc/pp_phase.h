// Phases of a layer: runs of consecutive gates that pp_phase.cu applies
// without a grid-wide barrier between them.
//
// A gate P mixes a string Q with Q xor P only.  So under a run of gates the
// strings fall into classes that never meet: Q's class is everything reached
// from Q by the run's generators.  When the run's gates commute pairwise, a
// gate that commutes with Q commutes with all of Q's class, so only the gates
// that anticommute with Q ("active" on its class) count.  A coarser label
// serves as well as the class itself, and a cheap one is the string with every
// bit that an active generator touches masked out.  For a run that does not
// commute pairwise the mask is that of all its generators.
//
// Plain C++ (no CUDA), so that the CPU tests can compile it.
#pragma once

#include <cmath>
#include <cstdint>
#include <vector>

namespace ppphase {

constexpr int kShortRun = 6;
constexpr int kMaxGates = 32;  // gates of a phase: one bit each in a 32-bit mask

struct Phase {
  int first = 0, count = 0;  // gates [first, first + count) in application order
  int commuting = 0;         // pairwise commuting: classes from the active gates
  int triangular = 0;        // and every generator has a bit that no later one has
  uint64_t ux[4] = {0, 0, 0, 0}, uz[4] = {0, 0, 0, 0};  // OR of the generators
};

// Generators of one gate, words [0, W).
struct Gen {
  const uint64_t* x;
  const uint64_t* z;
};

inline bool commute(const Gen& a, const Gen& b, int W) {
  int p = 0;
  for (int j = 0; j < W; ++j) p ^= __builtin_popcountll((a.x[j] & b.z[j]) ^ (a.z[j] & b.x[j])) & 1;
  return p == 0;
}

// Gates that some string may anticommute with (damp: or be damped by), from the
// OR of all strings' x and z words, widened by each such gate's letters as the
// kernels widen it.  The others leave every string as it is.
inline std::vector<unsigned char> touched(const std::vector<Gen>& gates, int W, const uint64_t* occ_x,
                                          const uint64_t* occ_z, bool damp) {
  uint64_t ox[4], oz[4];
  for (int j = 0; j < W; ++j) ox[j] = occ_x[j], oz[j] = occ_z[j];
  std::vector<unsigned char> out(gates.size(), 0);
  for (size_t g = 0; g < gates.size(); ++g) {
    const Gen& p = gates[g];
    uint64_t t = 0;
    for (int j = 0; j < W; ++j) {
      t |= (p.x[j] & oz[j]) | (p.z[j] & ox[j]);
      if (damp) t |= (p.x[j] | p.z[j]) & (ox[j] | oz[j]);
    }
    if (!t) continue;
    out[g] = 1;
    for (int j = 0; j < W; ++j) ox[j] |= p.x[j], oz[j] |= p.z[j];
  }
  return out;
}

// How a layer is cut.
struct Limits {
  int max_gates = kMaxGates;  // per phase
  int max_plain = kMaxGates;  // of commuting ones that are not triangular
  double max_active = 3.0;    // mean number of its gates active on a string
  int max_bits = 10;          // key bits a phase that does not commute may touch
  bool triangular = false;    // dense classes are possible: look for triangular runs
  size_t max_phases = ~(size_t)0;  // the plan stops at one more
};

// Cut the gates into phases, greedily.  Gates that touch nothing are in no
// phase, or between the gates of one.
//
// A run of commuting gates (up to the first that does not commute with all
// before it) is cut into equal parts in which at most max_active gates are active
// on a string on average (activity: per gate, from the layer before): classes grow
// with the number of active gates, and a class has to fit one block.
// With `triangular` a part also ends where a gate would leave an earlier one
// without a bit of its own.  Parts of fewer than kShortRun gates give way to a run
// whose generators touch at most max_bits key bits (at most 2^max_bits strings
// per class), if that is longer -- three times as long where the part would be
// dense, which is several times faster.
inline std::vector<Phase> plan(const std::vector<Gen>& gates, int W, const unsigned char* touch,
                               const float* activity, const Limits& lim) {
  std::vector<Phase> out;
  const int G = (int)gates.size();
  const int most[2] = {lim.max_plain < kMaxGates ? lim.max_plain : kMaxGates,
                       lim.max_gates < kMaxGates ? lim.max_gates : kMaxGates};
  int run_end = 0;        // of the commuting run that g is in
  double part_act = 0.0;  // activity of one of its parts
  for (int g = 0; g < G && out.size() <= lim.max_phases;) {
    if (!touch[g]) {
      ++g;
      continue;
    }
    if (g >= run_end) {
      double total = 0.0;
      int n = 0;
      run_end = g;
      for (; run_end < G && n < 96; ++run_end) {
        if (!touch[run_end]) continue;  // does nothing, wherever it stands
        bool ok = true;
        for (int k = g; k < run_end && ok; ++k)
          ok = !touch[k] || commute(gates[k], gates[run_end], W);
        if (!ok) break;
        total += activity[run_end];
        ++n;
      }
      const double parts = std::ceil(total / lim.max_active);
      part_act = parts > 1.0 ? total / parts : lim.max_active;
    }
    int c = g, nc = 0;  // end of the part, its gates that touch
    bool tri = lim.triangular;
    std::vector<uint64_t> own;  // bits of each generator that no later one has, [x, z][W]
    double act = 0.0;
    for (; c < run_end && c - g < kMaxGates; ++c) {
      if (!touch[c]) continue;
      if (nc >= most[tri] || (nc > 0 && act + 0.5 * activity[c] > part_act)) break;
      if (tri) {
        bool keeps = true;
        for (size_t k = 0; k < own.size() && keeps; k += 2 * W) {
          uint64_t left = 0;
          for (int j = 0; j < W; ++j)
            left |= (own[k + j] & ~gates[c].x[j]) | (own[k + W + j] & ~gates[c].z[j]);
          keeps = left != 0;
        }
        if (!keeps) {
          if (nc >= kShortRun) break;
          tri = false;
        } else {
          for (size_t k = 0; k < own.size(); k += 2 * W)
            for (int j = 0; j < W; ++j) {
              own[k + j] &= ~gates[c].x[j];
              own[k + W + j] &= ~gates[c].z[j];
            }
          for (int j = 0; j < W; ++j) own.push_back(gates[c].x[j]);
          for (int j = 0; j < W; ++j) own.push_back(gates[c].z[j]);
        }
      }
      act += activity[c];
      ++nc;
    }
    int e = g, ne = 0;  // end of the run with few bits, its gates that touch
    uint64_t ux[4] = {0, 0, 0, 0}, uz[4] = {0, 0, 0, 0};
    for (; nc < kShortRun && e < G && e - g < kMaxGates; ++e) {
      if (!touch[e]) continue;
      int bits = 0;
      for (int j = 0; j < W; ++j)
        bits += __builtin_popcountll(ux[j] | gates[e].x[j]) + __builtin_popcountll(uz[j] | gates[e].z[j]);
      if (bits > lim.max_bits) break;
      for (int j = 0; j < W; ++j) {
        ux[j] |= gates[e].x[j];
        uz[j] |= gates[e].z[j];
      }
      ++ne;
    }
    Phase p;
    p.first = g;
    p.commuting = nc >= kShortRun || ne <= (tri ? 3 : 1) * nc ? 1 : 0;
    p.triangular = p.commuting && tri;
    p.count = (p.commuting ? c : e) - g;
    const int next = g + p.count;
    while (!touch[g + p.count - 1]) --p.count;  // the first one touches
    for (int k = g; k < g + p.count; ++k)
      for (int j = 0; j < W && touch[k]; ++j) {
        p.ux[j] |= gates[k].x[j];
        p.uz[j] |= gates[k].z[j];
      }
    out.push_back(p);
    g = next;
    if (!p.commuting) run_end = g;  // the run it cut into starts anew
  }
  return out;
}

// Whether a layer's table is so full that its classes are too: most of the 2^r
// strings of a class are there, and the classes are few and uneven, a warp each.  On
// the persistent kernel then, unless all phases are dense (a block's sweep takes full
// classes best of all) or the table is small (a gate's barrier counts for more).
// All-to-all Heisenberg layers, phases and persistent kernel, us: 10 qubits, 262144
// strings (4^n / 4) 3120 and 1860; 12 qubits, 225 to 509 thousand (1.3 to 3 %) 5010
// and 3700, 75 to 225 thousand 2400 and 2390; 14 qubits, 190 to 644 thousand (1 %
// expected) 4220 and 4700; a 3 x 4 torus, 23 to 101 thousand (2.4 % expected), given up
// after 2500, 690; 8 qubits, 3280 to 16384 strings 680 and 890, 16384 to 16384
// 605 and 520; tori of 3 x 3, 12 to 25 thousand 910 and 530, 8590 to 9410 strings 220
// and 490.
constexpr uint64_t kFullTerms = 11000;
constexpr double kFullShare = 1.0 / 64;
inline bool nearly_full(uint64_t terms, double expected, int n, const std::vector<Phase>& phases) {
  if (terms < kFullTerms || expected < kFullShare * std::pow(4.0, n)) return false;
  for (const Phase& p : phases)
    if (!p.triangular) return true;
  return false;
}

// Buckets of one phase, and the records each has room for.
struct Room {
  uint64_t nb = 0, cg = 0;
};

// What takes a phase's buckets, a block or a warp each: how many strings one is to
// hold, and how many buckets keep the chip busy.
struct Workers {
  double fill;
  uint64_t least;
};

// Strings expected at the end of a layer, and what a bucket may meet of them.
struct Expected {
  double strings;  // that buckets are made for
  double lumps;    // the growth of the layer before, extrapolated
};

// The next growth is a quarter above the last one, as far as that goes: one term
// becomes thousands in the first layer of an all-to-all circuit, and the tables
// after it ten times as many each, not thousands of times.  (Buckets for all of the
// extrapolation: 4 GB for the 16384 strings of 8 qubits, 20 GB for 75 thousand of 12,
// whose counters a warp goes through one after the other.)  Nor are there more strings
// than the tables hold, which is `possible`.
constexpr double kMostGrowth = 32.0;
inline Expected expected(uint64_t terms, double last_growth, double possible) {
  const double grown = (double)terms * (1.25 * last_growth > 1.5 ? 1.25 * last_growth : 1.5);
  const double most = std::fmin((double)terms * kMostGrowth, possible);
  return {std::fmin(grown, most), grown};
}

// A bucket has room for four times its share and more, since classes come in lumps:
// up to four times `fill` where the table is growing fast.
inline Room bucket_room(const Expected& e, const Workers& w, double factor) {
  Room r;
  r.nb = (uint64_t)std::ceil(std::fmin(e.strings * factor / w.fill, 1e12));
  if (r.nb < w.least) r.nb = w.least;
  r.cg = (256 + (uint64_t)(4.0 * std::fmin(e.lumps / (double)w.least, w.fill / factor))) / 8 * 8;
  return r;
}

// Each phase's, by what takes its buckets.  (With the buckets of the blocks for all,
// all-to-all layers with truncation, whose phases are not dense, ran on 304 of 1824
// warps; with those of the warps for all, a dense phase takes many times the parts.)
inline std::vector<Room> bucket_rooms(const std::vector<Phase>& phases, const Expected& e, const Workers& dense,
                                      const Workers& sparse, double factor) {
  std::vector<Room> out;
  for (const Phase& p : phases) out.push_back(bucket_room(e, p.triangular ? dense : sparse, factor));
  return out;
}

}  // namespace ppphase
