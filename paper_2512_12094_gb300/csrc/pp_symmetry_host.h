// Symmetry groups on host-side Pauli strings (x words, then z words): the
// group codes, each group's generators as maps of sites, and the invariance
// tests pp_create and pp_apply_layer use to reject a layer, an observable or
// a state the declared group does not map onto itself (PP_ERR_SYMMETRY).
// Plain C++ with no CUDA, so the same code is compiled into the library and
// into a CPU test driver.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "../../include/pp.h"

namespace ppsym {

inline void permute_string(const uint64_t* x, const uint64_t* z, int W,
                           const std::vector<int>& to, uint64_t* ox, uint64_t* oz) {
  for (int j = 0; j < W; ++j) ox[j] = oz[j] = 0;
  for (int j = 0; j < W; ++j)  // the sites that hold a letter
    for (uint64_t m = x[j] | z[j]; m; m &= m - 1) {
      const int b = __builtin_ctzll(m), t = to[64 * j + b];
      ox[t >> 6] |= ((x[j] >> b) & 1ull) << (t & 63);
      oz[t >> 6] |= ((z[j] >> b) & 1ull) << (t & 63);
    }
}

// Group codes: kind in the low byte (pp_symmetry), torus width above it.
inline int group_kind(int code) { return code & 0xFF; }
inline int group_lx(int code) { return code >> 8; }

inline bool valid_group(int code, int n) {
  const int kind = group_kind(code), lx = group_lx(code);
  if (code < 0 || kind > PP_SYM_TORUS) return false;
  if (kind == PP_SYM_TORUS) return lx >= 1 && lx <= n && n % lx == 0;
  return lx == 0;
}

// Generators of the group as site maps (the letter of q moves to to[q]).
inline std::vector<std::vector<int>> generators(int group, int n) {
  std::vector<std::vector<int>> gens;
  const int kind = group_kind(group);
  if (n < 2 || kind == PP_SYM_NONE) return gens;
  if (kind == PP_SYM_TORUS) {
    const int lx = group_lx(group), ly = n / lx;
    std::vector<int> sx(n), sy(n);
    for (int q = 0; q < n; ++q) {
      const int x = q % lx, y = q / lx;
      sx[q] = (x + 1) % lx + lx * y;
      sy[q] = x + lx * ((y + 1) % ly);
    }
    gens.push_back(sx);
    gens.push_back(sy);
    return gens;
  }
  std::vector<int> shift(n);
  for (int q = 0; q < n; ++q) shift[q] = (q + n - 1) % n;  // T: qubit q -> q-1
  gens.push_back(shift);
  if (kind == PP_SYM_SN) {
    std::vector<int> swap01(n);
    for (int q = 0; q < n; ++q) swap01[q] = q;
    std::swap(swap01[0], swap01[1]);
    gens.push_back(swap01);
  }
  if (kind == PP_SYM_DN) {
    std::vector<int> refl(n);
    for (int q = 0; q < n; ++q) refl[q] = n - 1 - q;
    gens.push_back(refl);
  }
  return gens;
}

typedef std::vector<uint64_t> HKey;

// Positions of m keys of K words each in ascending order, equal keys in the
// order they came.
inline std::vector<uint32_t> key_order(const uint64_t* keys, size_t m, int K) {
  std::vector<uint32_t> at(m);
  for (size_t i = 0; i < m; ++i) at[i] = (uint32_t)i;
  std::sort(at.begin(), at.end(), [&](uint32_t a, uint32_t b) {
    const uint64_t *p = keys + (size_t)a * K, *q = keys + (size_t)b * K;
    for (int j = 0; j < K; ++j)
      if (p[j] != q[j]) return p[j] < q[j];
    return a < b;
  });
  return at;
}

// Is the multiset {(string_i, value_i)} mapped onto itself by every generator?
// keys: m strings, x words then z words.  Both sides are sorted by string and,
// within equal strings, by value, and compared place by place (a map of vectors
// took 1 us a string and generator).
inline bool multiset_invariant(int group, int n, int W, const uint64_t* keys, const double* vals,
                               size_t m, double rel_tol) {
  const int K = 2 * W;
  auto equal = [&](const uint64_t* p, const uint64_t* q) {
    for (int j = 0; j < K; ++j)
      if (p[j] != q[j]) return false;
    return true;
  };
  // values in the order of at, sorted within equal keys
  auto sorted_values = [&](const uint64_t* k, const std::vector<uint32_t>& at) {
    std::vector<double> v(m);
    for (size_t i = 0; i < m; ++i) v[i] = vals[at[i]];
    for (size_t i = 0; i < m;) {
      size_t e = i + 1;
      while (e < m && equal(k + (size_t)at[i] * K, k + (size_t)at[e] * K)) ++e;
      if (e - i > 1) std::sort(v.begin() + (long)i, v.begin() + (long)e);
      i = e;
    }
    return v;
  };
  const std::vector<std::vector<int>> gens = generators(group, n);
  if (gens.empty()) return true;
  const std::vector<uint32_t> base = key_order(keys, m, K);
  const std::vector<double> base_v = sorted_values(keys, base);
  std::vector<uint64_t> img(m * (size_t)K);
  for (const auto& g : gens) {
    for (size_t i = 0; i < m; ++i) {
      const uint64_t* k = keys + i * K;
      permute_string(k, k + W, W, g, &img[i * K], &img[i * K + W]);
    }
    const std::vector<uint32_t> at = key_order(img.data(), m, K);
    const std::vector<double> v = sorted_values(img.data(), at);
    for (size_t i = 0; i < m; ++i) {
      if (!equal(keys + (size_t)base[i] * K, &img[(size_t)at[i] * K])) return false;
      const double a = v[i], b = base_v[i];
      if (std::fabs(a - b) > rel_tol * std::max(1.0, std::max(std::fabs(a), std::fabs(b)))) return false;
    }
  }
  return true;
}

inline bool multiset_invariant(int group, int n, int W, const std::vector<HKey>& keys,
                               const std::vector<double>& vals, double rel_tol) {
  std::vector<uint64_t> flat;
  flat.reserve(keys.size() * 2 * W);
  for (const HKey& k : keys) flat.insert(flat.end(), k.begin(), k.end());
  return multiset_invariant(group, n, W, flat.data(), vals.data(), keys.size(), rel_tol);
}

inline bool bloch_invariant(int group, int n, const double* bloch) {
  for (const auto& g : generators(group, n))
    for (int q = 0; q < n; ++q)
      for (int a = 0; a < 3; ++a)
        if (bloch[3 * q + a] != bloch[3 * g[q] + a]) return false;
  return true;
}

}  // namespace ppsym
