// What the kernels of phases share (pp_phase.cu, pp_phase_rows.cu): strings in
// 32-bit words, their class in the phase that comes next, and the buckets.
#pragma once

#include "pp_device.cuh"

namespace ppk {
namespace {

// A block's bucket is cut into at most 2^kMaxSplit parts.  Two classes that only just fit a
// part each must not meet in one: with 10 bits they did in some bucket of thousands.
constexpr int kMaxSplit = 16;

template <int P>
struct alignas(P == 1 ? 8 : 16) PKey {
  uint32_t w[2 * P];  // x words, then z words
};

// Generators of the phase that comes next, and for a dense one a bit of each that
// no later one has (gates that touch no string left out).
template <int P>
struct NextGens {
  static constexpr int kPivots = P <= 2 ? kPhaseGates : 1;  // dense phases: P <= 2
  PKey<P> gen[kPhaseGates];
  PKey<P> pivot[kPivots];
};

// Odd when the generator and the string anticommute.
template <int P>
__device__ __forceinline__ int anti_parity(const uint32_t* p, const uint32_t* q) {
  uint32_t v = 0;
#pragma unroll
  for (int j = 0; j < P; ++j) v ^= (p[j] & q[P + j]) ^ (p[P + j] & q[j]);
  return __popc(v);
}

// A key of the table (64-bit words) in 32-bit words, and back.
template <int P>
__device__ __forceinline__ PKey<P> ld_table_key(const uint64_t* keys, uint64_t i) {
  constexpr int W = (P + 1) / 2;
  const Key<W> K = ld_key<W>(keys, i);
  PKey<P> r;
#pragma unroll
  for (int j = 0; j < P; ++j) {
    r.w[j] = (uint32_t)(K.x(j / 2) >> (32 * (j & 1)));
    r.w[P + j] = (uint32_t)(K.z(j / 2) >> (32 * (j & 1)));
  }
  return r;
}

template <int P>
__device__ __forceinline__ Key<(P + 1) / 2> table_key(const PKey<P>& k) {
  constexpr int W = (P + 1) / 2;
  Key<W> r;
#pragma unroll
  for (int j = 0; j < W; ++j) {
    r.x(j) = k.w[2 * j];
    r.z(j) = k.w[P + 2 * j];
    if (P > 1) {
      r.x(j) |= (uint64_t)k.w[2 * j + (P > 1)] << 32;
      r.z(j) |= (uint64_t)k.w[P + 2 * j + (P > 1)] << 32;
    }
  }
  return r;
}

template <int P>
__device__ __forceinline__ PKey<P> ld_pkey(const uint32_t* keys, uint64_t i) {
  PKey<P> r;
  if constexpr (P == 1) {
    const uint2 v = reinterpret_cast<const uint2*>(keys)[i];
    r.w[0] = v.x;
    r.w[1] = v.y;
  } else {
    const uint4* p = reinterpret_cast<const uint4*>(keys) + i * (P / 2);
#pragma unroll
    for (int j = 0; j < P / 2; ++j) {
      const uint4 v = p[j];
      r.w[4 * j] = v.x;
      r.w[4 * j + 1] = v.y;
      r.w[4 * j + 2] = v.z;
      r.w[4 * j + 3] = v.w;
    }
  }
  return r;
}

template <int P>
__device__ __forceinline__ void st_pkey(uint32_t* keys, uint64_t i, const PKey<P>& k) {
  if constexpr (P == 1) {
    reinterpret_cast<uint2*>(keys)[i] = make_uint2(k.w[0], k.w[1]);
  } else {
    uint4* p = reinterpret_cast<uint4*>(keys) + i * (P / 2);
#pragma unroll
    for (int j = 0; j < P / 2; ++j)
      p[j] = make_uint4(k.w[4 * j], k.w[4 * j + 1], k.w[4 * j + 2], k.w[4 * j + 3]);
  }
}

template <int P>
__device__ __forceinline__ uint64_t string_hash(const PKey<P>& v, uint32_t seed) {
  uint32_t a = 0x9E3779B9u ^ seed, b = 0x7F4A7C15u + seed;
#pragma unroll
  for (int j = 0; j < P; ++j) {
    const uint32_t lo = v.w[j], hi = v.w[P + j];
    a = (a ^ lo) * 0xcc9e2d51u;
    a = __funnelshift_l(a, a, 15) ^ hi;
    a *= 0x1b873593u;
    b = (b ^ hi) * 0x27d4eb2fu;
    b = __funnelshift_l(b, b, 13) ^ lo;
    b *= 0x165667b1u;
  }
  return ((uint64_t)fmix32(a ^ b) << 32) | fmix32(b + 0x9E3779B9u * a);
}

// Active gates and class hash of a string in the phase that comes next: the hash
// of the string with the bits masked out that an active generator touches, or,
// for a dense phase, of the string reduced by its active generators (where it
// has the pivot of one, that one is taken out), which names the class exactly.
template <int P>
__device__ __forceinline__ void classify(const PKey<P>& K, const NextGens<P>& next,
                                         const PhaseDesc& d, unsigned& act, uint64_t& h) {
  PKey<P> v = K;
  act = 0;
  if (P <= 2 && d.dense) {
#pragma unroll 4
    for (int g = 0; g < d.count; ++g) {
      const PKey<P> G = next.gen[g], V = next.pivot[P <= 2 ? g : 0];
      const uint32_t on = 0u - (uint32_t)(anti_parity<P>(G.w, K.w) & 1);
      act |= on & (1u << g);
      uint32_t t = 0;
#pragma unroll
      for (int j = 0; j < 2 * P; ++j) t |= v.w[j] & V.w[j];
      const uint32_t out = t ? on : 0u;
#pragma unroll
      for (int j = 0; j < 2 * P; ++j) v.w[j] ^= G.w[j] & out;
    }
  } else if (d.commuting) {
    PKey<P> m;  // bits to mask out
#pragma unroll
    for (int j = 0; j < 2 * P; ++j) m.w[j] = 0;
#pragma unroll 4
    for (int g = 0; g < d.count; ++g) {
      const PKey<P> G = next.gen[g];
      const uint32_t on = 0u - (uint32_t)(anti_parity<P>(G.w, K.w) & 1);
      act |= on & (1u << g);
#pragma unroll
      for (int j = 0; j < 2 * P; ++j) m.w[j] |= G.w[j] & on;
    }
#pragma unroll
    for (int j = 0; j < 2 * P; ++j) v.w[j] &= ~m.w[j];
  } else {
#pragma unroll
    for (int j = 0; j < P; ++j) {
      v.w[j] &= ~(uint32_t)(d.ux[j / 2] >> (32 * (j & 1)));
      v.w[P + j] &= ~(uint32_t)(d.uz[j / 2] >> (32 * (j & 1)));
    }
  }
  h = string_hash<P>(v, act);
}

template <int P>
constexpr int kRecord = 1 + (P + 1) / 2;  // units of a bucket's record

// Append a string to its bucket of the next phase.
template <int P>
__device__ __forceinline__ void deal(const PhaseBuckets& out, const PKey<P>& K, double c, unsigned act,
                                     uint64_t h, unsigned& fail) {
  const unsigned b = (unsigned)(((h >> 32) * (uint64_t)out.nb) >> 32);
  const unsigned p = atomicAdd(out.cnt + b, 1u);
  if (p < out.cg) {
    const uint64_t at = (uint64_t)b * out.cg + p;
    uint4* const r = out.rec + at * kRecord<P>;
    r[0] = make_uint4((unsigned)__double2loint(c), (unsigned)__double2hiint(c), act, (unsigned)h);
    st_pkey<P>(reinterpret_cast<uint32_t*>(r + 1), 0, K);
  } else {
    fail |= kPhaseBucketFull;
  }
}

// All threads of the block; ends with a barrier.
template <int P>
__device__ __forceinline__ void load_generators(NextGens<P>& to, const GateArgs* gates, const PhaseDesc& d) {
  for (int k = threadIdx.x; k < d.count * 2 * P; k += blockDim.x) {
    const int g = k / (2 * P), j = k % (2 * P), q = j % P;
    const uint64_t* src = j < P ? gates[d.first + g].px : gates[d.first + g].pz;
    to.gen[g].w[j] = (uint32_t)(src[q / 2] >> (32 * (q & 1)));
  }
  __syncthreads();
  if (P <= 2 && d.dense) {
    for (int g = threadIdx.x; g < d.count; g += blockDim.x) {
      PKey<P> own = to.gen[g];
      for (int k = g + 1; k < d.count; ++k)
        if (!((d.skip >> k) & 1u)) {
#pragma unroll
          for (int j = 0; j < 2 * P; ++j) own.w[j] &= ~to.gen[k].w[j];
        }
      bool first = true;  // its lowest bit
#pragma unroll
      for (int j = 0; j < 2 * P; ++j) {
        const uint32_t bit = first ? own.w[j] & (0u - own.w[j]) : 0u;
        if (bit) first = false;
        to.pivot[P <= 2 ? g : 0].w[j] = bit;
      }
    }
    __syncthreads();
  }
}

constexpr int kDRank = kPhaseRank;
constexpr unsigned kSample = 8;  // buckets whose strings are counted per gate: one in so many

// A key in P 64-bit words: x | z << 32 (P = 1), or x, z (P = 2).
template <int P>
struct DKey {
  uint64_t a[P];
};

template <int P>
__device__ __forceinline__ DKey<P> pack_key(const PKey<P>& k) {
  DKey<P> r;
  if constexpr (P == 1) {
    r.a[0] = k.w[0] | ((uint64_t)k.w[1] << 32);
  } else {
    r.a[0] = k.w[0] | ((uint64_t)k.w[1] << 32);
    r.a[1] = k.w[2] | ((uint64_t)k.w[3] << 32);
  }
  return r;
}

template <int P>
__device__ __forceinline__ PKey<P> unpack_pkey(const DKey<P>& k) {
  PKey<P> r;
  r.w[0] = (uint32_t)k.a[0];
  r.w[1] = (uint32_t)(k.a[0] >> 32);
  if constexpr (P == 2) {
    r.w[2] = (uint32_t)k.a[1];
    r.w[3] = (uint32_t)(k.a[1] >> 32);
  }
  return r;
}

template <int P>
__device__ __forceinline__ uint64_t x_of(const DKey<P>& k) { return P == 1 ? (k.a[0] & 0xFFFFFFFFull) : k.a[0]; }
template <int P>
__device__ __forceinline__ uint64_t z_of(const DKey<P>& k) { return P == 1 ? (k.a[0] >> 32) : k.a[P - 1]; }

template <int P>
struct DGate {
  DKey<P> p;
  DKey<P> pivot;  // a bit of p that no later generator of the phase has
  double cth, sth;
  int pyy;
  int after, skip_after;  // gates of the layer after this one; those that touch nothing
};

template <int P>
__device__ __forceinline__ unsigned table_slot(const DKey<P>& k) {
  uint64_t h = k.a[0] * 0x9E3779B97F4A7C15ull;
  if constexpr (P == 2) h = (h ^ (h >> 29) ^ k.a[1]) * 0xBF58476D1CE4E5B9ull;
  h ^= h >> 32;
  return (unsigned)(h * 0x94D049BB133111EBull >> 53);  // kDTable = 2^11
}

// i P Q = -R for the gate and the string at a slot.
template <int P>
__device__ __forceinline__ bool child_negative(const DGate<P>& G, const DKey<P>& Q, const DKey<P>& R) {
  int e = G.pyy;
  if constexpr (P == 1) {
    const uint32_t qx = (uint32_t)Q.a[0], qz = (uint32_t)(Q.a[0] >> 32);
    const uint32_t rx = (uint32_t)R.a[0], rz = (uint32_t)(R.a[0] >> 32);
    e += __popc(qx & qz) - __popc(rx & rz) + 2 * __popc((uint32_t)(G.p.a[0] >> 32) & qx);
  } else {
    e += __popcll(Q.a[0] & Q.a[P - 1]) - __popcll(R.a[0] & R.a[P - 1]) +
         2 * __popcll(G.p.a[P - 1] & Q.a[0]);
  }
  return ((e + 1) & 3) != 0;
}

}  // namespace
}  // namespace ppk
