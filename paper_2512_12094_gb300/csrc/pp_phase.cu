// A layer as a few phases (pp_phase.h) instead of one grid-wide pass per gate.
//
// Before a phase the strings are dealt into buckets by the hash of their
// class; a warp then takes a bucket into its share of the block's shared memory
// and applies all the phase's gates there, partners found in a small hash index
// in shared memory, and deals the surviving strings into the buckets of the
// next phase (after the last one: into a dense table).  The arithmetic per pair
// is that of gate_pass, so the table is the same bit for bit; no string of
// another warp is ever needed, so nothing waits on the grid or on the block,
// and the table needs no index in global memory.
//
// Why: one pass per gate costs a grid barrier, dependent L2 loads and a births
// flush whatever the table (9 us a gate at 10^5 strings), and three random
// 32-byte HBM sectors per anticommuting string on large tables.  A phase costs
// two passes over the table (a record of 32 bytes a string in and out up to 64 sites,
// half of it scattered) and the instructions of the gates, which are what bounds it.
//
// Why a warp per bucket: only some 15 % of a bucket's strings anticommute with
// a gate.  A warp needs 200 strings or more to fill its lanes with them; blocks
// of 8 warps on a bucket of 250 strings ran 160 instructions per string and
// phase at 14 % of the FP64 lanes and waited at a barrier per gate.
//
// A bucket that outgrows the warp is done again in parts, split by further
// bits of the class hash; a class that outgrows it, a full bucket or a full
// destination sets PhaseStat::fail.  The layer's input table is never written,
// so the host then applies the layer by the other path.
#include <algorithm>

#include "pp_phase.cuh"
#include "pp_smem_limit.h"

namespace ppk {
namespace {

constexpr int kPW = 4;          // warps of a phase block
constexpr int kPT = 32 * kPW;
// A warp's bucket is cut into at most 2^kWarpSplit parts (a class that is too large
// among small ones is found by cutting on: 85 us a bit at 4 words, 16 bits 2.3 ms of a
// layer given up and 10 bits 1.7)
constexpr int kWarpSplit = 10;
constexpr int kPosBits = 11;    // of an index slot: position + 1; a tag above it
constexpr unsigned kPosMask = (1u << kPosBits) - 1u;
// Strings are kept in P 32-bit words per plane: one for n <= 32 (half the
// shared memory and bucket traffic of the 64-bit words of the table).
// C: strings of a warp; kSlots: its index slots, at most 3/4 full.
template <int P>
struct PhaseDims {
  static constexpr int C = P == 1 ? 736 : (P == 2 ? 480 : (P == 4 ? 320 : (P == 6 ? 224 : 192)));
  static constexpr int kSlots = P == 1 ? 2048 : (P <= 4 ? 1024 : 512);
  static constexpr int kLoads = P <= 2 ? 4 : 2;  // strings a lane loads at once
};
constexpr int kPBlocks = 3;  // phase blocks an SM's shared memory holds

template <int P>
struct PGate {
  uint32_t p[2 * P];
  double cth, sth;
  uint32_t pvm;  // pivot bit
  int pvw;       // its word
  int pyy;
};

// A warp's bucket in shared memory.
template <int P>
struct PhaseWarp {
  static constexpr int C = PhaseDims<P>::C, kSlots = PhaseDims<P>::kSlots;
  PKey<P> key[C];
  double coef[C];
  uint16_t slot[kSlots];  // index: tag and position + 1; 0 = empty
  uint16_t list[64];
  int acdl[kPhaseGates];  // live anticommuting strings << 16, plus the live change
};

template <int P>
struct PhaseSmem {
  PhaseWarp<P> warp[kPW];
  PGate<P> gate[kPhaseGates];
  NextGens<P> next;
  unsigned long long ac[kPhaseGates];
  long long dl[kPhaseGates];
};

// Hash of a key for the index, its first slot and its tag.
template <int P>
__device__ __forceinline__ uint32_t index_hash(const PKey<P>& k) {
  uint32_t h = 0;
#pragma unroll
  for (int j = 0; j < 2 * P; ++j) h = (h ^ k.w[j]) * 0x9E3779B1u + (h >> 15);
  h ^= h >> 16;
  return h * 0x85ebca6bu;
}
template <int S>
__device__ __forceinline__ unsigned first_slot(uint32_t h) {
  return (unsigned)(((uint64_t)h * S) >> 32);
}
__device__ __forceinline__ unsigned slot_tag(uint32_t h) { return (h << kPosBits) & 0xFFFFu; }

template <int P>
__device__ __forceinline__ int y_count(const uint32_t* w) {
  int y = 0;
#pragma unroll
  for (int j = 0; j < P; ++j) y += __popc(w[j] & w[P + j]);
  return y;
}

// Clear the layer's counters (cleared words follow the PhaseStat) and reset the
// context's append cursor, occupancy masks and stall flag.
__global__ void __launch_bounds__(kBlock)
    phase_begin_kernel(unsigned* words, uint64_t n, DevCtl* ctl) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) words[i] = 0u;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctl->n_next = 0;
    ctl->stall = 0;
    for (int j = 0; j < 2 * kMaxW; ++j) ctl->occ[j] = 0ull;
  }
}

// Live entries of a dense table into the buckets of the first phase.
template <int P>
__global__ void __launch_bounds__(kBlock)
    phase_deal_kernel(const uint64_t* __restrict__ keys, const double* __restrict__ coef, uint64_t T,
                      int use_eps, PhaseBuckets out, PhaseDesc d,
                      const GateArgs* __restrict__ gates, PhaseAcc acc) {
  __shared__ __align__(16) NextGens<P> next;
  __shared__ unsigned s_live;
  if (threadIdx.x == 0) s_live = 0;
  load_generators<P>(next, gates, d);
  unsigned fail = 0, live = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < T; i += stride) {
    const double c = coef[i];
    const PKey<P> K = ld_table_key<P>(keys, i);
    if (use_eps && is_zero_bits(c)) continue;
    ++live;
    unsigned act;
    uint64_t h;
    classify<P>(K, next, d, act, h);
    deal<P>(out, K, c, act, h, fail);
  }
  live = __reduce_add_sync(kFull, live);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_live, live);
  if (fail) atomicOr(&acc.st->fail, fail);
  __syncthreads();
  if (threadIdx.x == 0 && s_live) atomicAdd(&acc.st->live0, (unsigned long long)s_live);
}

// Claim an index slot for the string at position p (one warp writes the index).
template <int S>
__device__ __forceinline__ void claim_slot(uint16_t (&slot)[S], uint32_t h, int p) {
  const unsigned short v = (unsigned short)(slot_tag(h) | (unsigned)(p + 1));
  unsigned pos = first_slot<S>(h);
  while (atomicCAS(&slot[pos], (unsigned short)0, v) != 0) pos = (pos + 1) & (S - 1);
}

// The gates of a phase over the n strings of a warp; the new count, or -1 when
// births pass the warp's room.
template <int P>
__device__ __forceinline__ int phase_gates(PhaseWarp<P>& S, const PGate<P>* gates,
                                           const PhaseDesc& d, const PhaseRule& rule, int n,
                                           unsigned uni) {
  constexpr int C = PhaseWarp<P>::C, kSlots = PhaseWarp<P>::kSlots;
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const bool use_eps = rule.use_eps != 0;
  const uint64_t eps_bits = rule.eps_bits;
  const double* damp = rule.damp;
  auto is_dead = [&](double c) { return use_eps && is_zero_bits(c); };
  auto trunc = [&](double c) { return (use_eps && (dbits(c) & kAbsMask) < eps_bits) ? 0.0 : c; };
  // gates that are active on some string (damping needs them all)
  unsigned todo = n > 0 ? (d.count == 32 ? ~0u : ((1u << d.count) - 1u)) : 0u;
  if (d.commuting && !damp) todo &= uni;
  for (; todo; todo &= todo - 1) {
    const int g = __ffs(todo) - 1;
    const PGate<P>& G = gates[g];
    int delta = 0, n_ac = 0;
    int nn = n;  // with the births so far
    // one anticommuting string per lane
    auto work = [&](int k) {
      bool want = false;
      double child = 0.0;
      PKey<P> R;
      uint32_t h = 0;
      if (lane < k) {
        const int i = S.list[lane];
        const PKey<P> Q = S.key[i];
        const double cQ = S.coef[i];
        const bool liveQ = !is_dead(cQ);
#pragma unroll
        for (int j = 0; j < 2 * P; ++j) R.w[j] = Q.w[j] ^ G.p[j];
        // the member of {Q, R} with the pivot bit of P clear owns the pair
        const bool owner = (S.key[i].w[G.pvw] & G.pvm) == 0;
        h = index_hash<P>(R);
        int jr = -1;
        if (owner || liveQ) {  // a truncated string that owns nothing has nothing to do
          const unsigned tag = slot_tag(h);
          for (unsigned pos = first_slot<kSlots>(h);; pos = (pos + 1) & (kSlots - 1)) {
            const unsigned v = S.slot[pos];
            if (v == 0) break;
            const int s = (int)(v & kPosMask);
            if ((v & ~kPosMask) == tag && s <= n) {  // births of this gate are nobody's partner
              const PKey<P> K = S.key[s - 1];
              bool eq = true;
#pragma unroll
              for (int j = 0; j < 2 * P; ++j) eq &= K.w[j] == R.w[j];
              if (eq) {
                jr = s - 1;
                break;
              }
            }
          }
        }
        const double cR = (jr >= 0 && owner) ? S.coef[jr] : 0.0;
        const bool liveR = jr >= 0 && owner && !is_dead(cR);
        const bool birth = jr < 0 && liveQ;
        const bool own = owner && jr >= 0 && (liveQ || liveR);
        n_ac += birth ? 1 : (own ? (int)liveQ + (int)liveR : 0);
        if (own || birth) {
          // i P Q = i^{E+1} R (see sigma_of): from the Y counts of Q and R
          int e = G.pyy + y_count<P>(Q.w) - y_count<P>(R.w);
#pragma unroll
          for (int j = 0; j < P; ++j) e += 2 * __popc(G.p[P + j] & Q.w[j]);
          const bool neg = ((e + 1) & 3) != 0;
          double dQ = cQ, dR = cR;
          if (damp) {
            int kq = 0, kr = 0;
#pragma unroll
            for (int j = 0; j < P; ++j) {
              const uint32_t supp = G.p[j] | G.p[P + j];
              kq += __popc((Q.w[j] | Q.w[P + j]) & supp);
              kr += __popc((R.w[j] | R.w[P + j]) & supp);
            }
            if (kq) dQ = __dmul_rn(dQ, damp[kq]);
            if (own && kr) dR = __dmul_rn(dR, damp[kr]);
          }
          const double aQ = __dmul_rn(G.cth, dQ);
          const double sQ = __dmul_rn(G.sth, dQ);
          double nQ = aQ;
          if (own) {
            const double aR = __dmul_rn(G.cth, dR);
            const double sR = __dmul_rn(G.sth, dR);
            nQ = __dadd_rn(aQ, with_sign(sR, !neg));
            const double nR = trunc(__dadd_rn(aR, with_sign(sQ, neg)));
            S.coef[jr] = nR;
            delta += (int)!is_dead(nR) - (int)liveR;
          } else {
            child = with_sign(sQ, neg);
            int w = 0;
#pragma unroll
            for (int j = 0; j < P; ++j) w += __popc(R.w[j] | R.w[P + j]);
            want = (rule.wmax < 0 || w <= rule.wmax) &&
                   !(use_eps && (dbits(child) & kAbsMask) < eps_bits);
          }
          nQ = trunc(nQ);
          S.coef[i] = nQ;
          delta += (int)!is_dead(nQ) - (int)liveQ;
        }
      }
      const unsigned bal = __ballot_sync(kFull, want);
      if (want) {
        const int p = nn + __popc(bal & below);
        if (p < C) {
          S.key[p] = R;
          S.coef[p] = child;
          claim_slot(S.slot, h, p);
        }
        ++delta;
      }
      nn += __popc(bal);
    };
    int fill = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
      const int i = i0 + lane;
      bool a = false;
      if (i < n) {
        const PKey<P> K = S.key[i];
        a = anti_parity<P>(G.p, K.w) & 1;
        if (damp && !a) {
          int kq = 0;
#pragma unroll
          for (int j = 0; j < P; ++j) kq += __popc((K.w[j] | K.w[P + j]) & (G.p[j] | G.p[P + j]));
          if (kq) {
            const double c = S.coef[i];
            if (!is_dead(c)) {
              const double v = trunc(__dmul_rn(c, damp[kq]));
              delta -= (int)is_dead(v);
              S.coef[i] = v;
            }
          }
        }
      }
      const unsigned bal = __ballot_sync(kFull, a);
      if (a) S.list[fill + __popc(bal & below)] = (uint16_t)i;
      fill += __popc(bal);
      if (fill >= 32) {
        __syncwarp();
        work(32);
        __syncwarp();
        uint16_t v = 0;
        if (lane < fill - 32) v = S.list[32 + lane];
        __syncwarp();
        if (lane < fill - 32) S.list[lane] = v;
        fill -= 32;
      }
    }
    __syncwarp();
    if (fill) {
      work(fill);
      __syncwarp();
    }
    const int sum = __reduce_add_sync(kFull, n_ac * 65536 + delta);
    if (lane == 0) S.acdl[g] += sum;
    n = nn;
    if (n > C) return -1;
  }
  __syncwarp();
  return n;
}

// One phase: warp w of the grid takes buckets w, w + (warps), ... and deals what
// survives into the next phase's buckets, or (next.count == 0) appends it to
// the dense table `dense`.
template <int P>
__global__ void __launch_bounds__(kPT, kPBlocks)
    phase_kernel(PhaseBuckets in, PhaseBuckets out, PhaseDesc d,
                 PhaseDesc next, const GateArgs* __restrict__ gates, PhaseRule rule, DevTable dense,
                 DevCtl* ctl, PhaseAcc acc) {
  extern __shared__ __align__(16) unsigned char phase_raw[];
  PhaseSmem<P>& B = *reinterpret_cast<PhaseSmem<P>*>(phase_raw);
  constexpr int C = PhaseWarp<P>::C, kSlots = PhaseWarp<P>::kSlots;
  constexpr int W = (P + 1) / 2;
  // set by an earlier kernel of the stream, or by this one: then nothing of the
  // layer is kept
  if (__syncthreads_or(*reinterpret_cast<const volatile unsigned*>(&acc.st->fail) != 0u)) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned below = (1u << lane) - 1u;
  PhaseWarp<P>& S = B.warp[tid / 32];
  if (tid < d.count) {
    const GateArgs& a = gates[d.first + tid];
    PGate<P>& G = B.gate[tid];
    G.pvm = 0;
    G.pvw = 0;
#pragma unroll
    for (int j = 0; j < P; ++j) {
      G.p[j] = (uint32_t)(a.px[j / 2] >> (32 * (j & 1)));
      G.p[P + j] = (uint32_t)(a.pz[j / 2] >> (32 * (j & 1)));
      const uint32_t vx = (uint32_t)(a.pvx[j / 2] >> (32 * (j & 1)));
      const uint32_t vz = (uint32_t)(a.pvz[j / 2] >> (32 * (j & 1)));
      if (vx) G.pvm = vx, G.pvw = j;
      if (vz) G.pvm = vz, G.pvw = P + j;
    }
    G.cth = a.cth;
    G.sth = a.sth;
    G.pyy = a.pyy;
  }
  if (tid < kPhaseGates) {
    B.ac[tid] = 0;
    B.dl[tid] = 0;
  }
  load_generators<P>(B.next, gates, next);
  unsigned fail = 0;
  OccAcc<W> occ;
  const unsigned warps = gridDim.x * (kPW);
  // State of the warp: bucket b, of which it has the strings whose class hash
  // has the low s bits `id` in hand; s0 leaves room for births.
  unsigned b = blockIdx.x * (kPW) + tid / 32, id = 0;
  int cnt = 0, s = 0, s0 = 0;
  uint64_t base = 0;
  auto open = [&]() {  // the next bucket that holds anything
    cnt = 0;
    for (; b < in.nb; b += warps) {
      cnt = (int)min(in.cnt[b], in.cg);
      if (cnt) break;
    }
    base = (uint64_t)b * in.cg;
    s0 = 0;
    while ((cnt >> s0) > C * 3 / 4) ++s0;
    s = s0;
    id = 0;
  };
  open();
  while (cnt) {
    __syncwarp();
    for (int k = lane; k < kSlots / 2; k += 32) reinterpret_cast<unsigned*>(S.slot)[k] = 0u;
    for (int k = lane; k < kPhaseGates; k += 32) S.acdl[k] = 0;
    __syncwarp();
    unsigned uni = 0, all = ~0u, any = 0;
    int n = 0;
    constexpr int U = PhaseDims<P>::kLoads;
    for (int i0 = 0; i0 < cnt; i0 += 32 * U) {
      PKey<P> K[U];
      double c[U];
      uint2 m[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + 32 * u + lane;
        if (i < cnt) {
          const uint4* r = in.rec + (base + i) * kRecord<P>;
          const uint4 a = r[0];
          m[u] = make_uint2(a.z, a.w);
          K[u] = ld_pkey<P>(reinterpret_cast<const uint32_t*>(r + 1), 0);
          c[u] = __hiloint2double((int)a.y, (int)a.x);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + 32 * u + lane;
        const bool mine = i < cnt && (m[u].y & ((1u << s) - 1u)) == id;
        const unsigned bal = __ballot_sync(kFull, mine);
        const int p = n + __popc(bal & below);
        n += __popc(bal);
        if (mine) {
          uni |= m[u].x;
          all &= m[u].y;
          any |= m[u].y;
          if (p < C) {
            S.key[p] = K[u];
            S.coef[p] = c[u];
            claim_slot(S.slot, index_hash<P>(K[u]), p);
          }
        }
      }
    }
    uni = __reduce_or_sync(kFull, uni);
    __syncwarp();
    const bool too_many = n > C;
    // one class, which no further bit of its hash divides
    if (too_many && __reduce_and_sync(kFull, all) == __reduce_or_sync(kFull, any)) s = kWarpSplit;
    n = phase_gates<P>(S, B.gate, d, rule, too_many ? 0 : n, uni);
    if (too_many) n = -1;
    const bool ok = n >= 0;
    if (ok)
      for (int k = lane; k < d.count; k += 32) {
        const int v = S.acdl[k];
        if (v) {
          const int dl = (int)(short)(v & 0xFFFF);
          atomicAdd(&B.ac[k], (unsigned long long)((v - dl) >> 16));
          if (dl) atomicAdd(reinterpret_cast<unsigned long long*>(&B.dl[k]), (unsigned long long)(long long)dl);
        }
      }
    if (next.count) {
      for (int i = lane; i < n; i += 32) {
        const double c = S.coef[i];
        if (rule.use_eps && is_zero_bits(c)) continue;
        const PKey<P> K = S.key[i];
        unsigned act;
        uint64_t h;
        classify<P>(K, B.next, next, act, h);
        deal<P>(out, K, c, act, h, fail);
      }
    } else {
      // one reservation per part
      int kept = 0;
      for (int i = lane; i < n; i += 32) kept += !(rule.use_eps && is_zero_bits(S.coef[i]));
      int x = kept;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
      }
      unsigned long long at = 0;
      if (lane == 31 && x) at = atomicAdd(&ctl->n_next, (unsigned long long)x);
      at = __shfl_sync(kFull, at, 31) + (unsigned)(x - kept);
      for (int i = lane; i < n; i += 32) {
        const double c = S.coef[i];
        if (rule.use_eps && is_zero_bits(c)) continue;
        if (at < dense.cap) {
          const Key<W> K = table_key<P>(S.key[i]);
          st_key<W>(dense.keys, at, K);
          dense.coef[at] = c;
          occ.add(K);
        } else {
          fail |= kPhaseTableFull;
        }
        ++at;
      }
    }
    if (cnt) {
      if (!ok) {
        if (++s > kWarpSplit) {
          fail |= d.commuting ? kPhasePlainFull : kPhaseClassFull;
          cnt = 0;  // given up
        }
      } else {
        // the next part: up past the finished halves, then to the sibling
        while (s > 0 && ((id >> (s - 1)) & 1u)) {
          id &= ~(1u << (s - 1));
          --s;
        }
        if (s == 0) {
          b += warps;
          open();
        } else {
          id |= 1u << (s - 1);
          if (s < s0) s = s0;
        }
      }
    }
  }
  if (next.count == 0) occ.flush(ctl);
  if (fail) atomicOr(&acc.st->fail, fail);
  __syncthreads();
  if (tid < d.count) {
    const int g = d.first + tid;
    if (B.dl[tid])
      atomicAdd(reinterpret_cast<unsigned long long*>(acc.delta + g), (unsigned long long)B.dl[tid]);
    if (B.ac[tid]) atomicAdd(acc.ac + g, B.ac[tid]);
    if (blockIdx.x == 0 && !((d.skip >> tid) & 1u)) acc.touch[g] = 1u;
  }
}

// ------------------------------------------------------------ dense phases
//
// A phase of commuting gates with truncation on, strings of up to 64 qubits, each
// generator with a bit that no later one of the phase has.  A class of r active
// gates then has 2^r members, and once it has grown many of them are there.  So
// a block lays the classes of its bucket out as dense arrays of coefficients
// (absent = 0), bit k of a string's place saying whether the k-th active
// generator is in it, and a gate is a sweep over the pairs (j, j + 2^k) of all
// classes at once: no lookups, no births to place, full lanes, and a large class
// is spread over the block.  The
// FP64 pipe bounds it (24 cycles per warp instruction and SM, 6 a pair), where
// the sparse sweep above runs 300 instructions for every 32 anticommuting
// strings and waits for the one warp that has the largest class.

constexpr int kDT = 512;       // threads of a dense block
constexpr int kDStrings = 1024;
constexpr int kDSlots = 2048;  // coefficients of all classes of a part
// (class, active gate) entries: r for a class of 2^(r - 1) >= r pairs
constexpr int kDOrder = kDSlots / 2;
constexpr int kDTable = 2048;  // hash slots of the class lookup
struct DClass {
  uint16_t off, pairs;  // first slot, first pair
  uint16_t order;       // first of its active gates in DenseSmem::order
  uint16_t rank;        // active gates: 2^rank slots
};

template <int P>
struct DenseSmem {
  static_assert(2 * kDStrings >= kDSlots, "the survivors' list takes the place of act");
  DKey<P> slot_key[kDSlots];
  double slot[kDSlots];
  DKey<P> key[kDStrings];  // string, then the base of its class
  double coef[kDStrings];
  DGate<P> gate[kPhaseGates];
  NextGens<P> mine, next;
  DClass cls[kDStrings];
  uint32_t act[kDStrings];
  uint16_t coord[kDStrings];
  uint16_t member[kDStrings];    // the string that stands for the class
  uint16_t cid[kDStrings];       // class of a standing string
  uint16_t stand[kDStrings];     // standing string of a class
  uint16_t table[kDTable];       // position of a standing string + 1
  uint16_t pair_cls[kDSlots / 2];
  uint8_t order[kDOrder];        // active gates of the classes
  int bin[kDRank + 2];           // pairs per rank; then the first pair of the rank
  int upto[kDRank + 2];          // pairs of the classes of more than k active gates
  int n, slots, orders, classes, bad;
  unsigned out_n;
  unsigned long long out_base;
  unsigned seen[kPhaseGates];
};

template <int P>
__global__ void __launch_bounds__(kDT, 2)
    dense_phase_kernel(PhaseBuckets in, PhaseBuckets out, PhaseDesc d,
                       PhaseDesc next, const GateArgs* __restrict__ gates, PhaseRule rule,
                       DevTable dense, DevCtl* ctl, PhaseAcc acc) {
  extern __shared__ __align__(16) unsigned char phase_raw[];
  DenseSmem<P>& S = *reinterpret_cast<DenseSmem<P>*>(phase_raw);
  if (__syncthreads_or(*reinterpret_cast<const volatile unsigned*>(&acc.st->fail) != 0u)) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned below = (1u << lane) - 1u;
  const uint64_t eps_bits = rule.eps_bits;
  load_generators<P>(S.mine, gates, d);
  load_generators<P>(S.next, gates, next);
  if (tid < d.count) {
    const GateArgs& a = gates[d.first + tid];
    DGate<P>& G = S.gate[tid];
    if constexpr (P == 1) {
      G.p.a[0] = (a.px[0] & 0xFFFFFFFFull) | (a.pz[0] << 32);
    } else {
      G.p.a[0] = a.px[0];
      G.p.a[P - 1] = a.pz[0];
    }
    G.pivot = pack_key<P>(S.mine.pivot[tid]);
    G.cth = a.cth;
    G.sth = a.sth;
    G.pyy = a.pyy;
    G.after = d.after + d.count - 1 - tid;
    G.skip_after = d.skip_after + (tid + 1 < 32 ? __popc(d.skip >> (tid + 1)) : 0);
  }
  if (tid < kPhaseGates) S.seen[tid] = 0;
  unsigned fail = 0;
  long long upd = 0, skipped = 0;
  unsigned long long n_ac = 0;
  OccAcc<1> occ;
  for (unsigned b = blockIdx.x; b < in.nb; b += gridDim.x) {
    const int cnt = (int)min(in.cnt[b], in.cg);
    if (cnt == 0) continue;
    const uint64_t base = (uint64_t)b * in.cg;
    // parts of the bucket, as in phase_kernel
    int s0 = 0;
    while ((cnt >> s0) > kDStrings * 3 / 4) ++s0;
    int s = s0;
    unsigned id = 0;
    for (;;) {
      __syncthreads();  // the last part's readers are done
      for (int k = tid; k < kDTable / 2; k += kDT) reinterpret_cast<unsigned*>(S.table)[k] = 0u;
      if (tid == 0) {
        S.n = S.slots = S.orders = S.classes = S.bad = 0;
        S.out_n = 0;
      }
      if (tid < kDRank + 2) S.bin[tid] = 0;
      __syncthreads();
      for (int i0 = 0; i0 < cnt; i0 += kDT) {
        const int i = i0 + tid;
        const uint4* r = in.rec + (base + i) * kRecord<P>;
        uint4 a = make_uint4(0u, 0u, 0u, 0u);
        if (i < cnt) a = r[0];
        const bool mine = i < cnt && (a.w & ((1u << s) - 1u)) == id;
        const unsigned bal = __ballot_sync(kFull, mine);
        int p = 0;
        if (lane == 0 && bal) p = atomicAdd(&S.n, __popc(bal));
        p = __shfl_sync(kFull, p, 0) + __popc(bal & below);
        if (mine && p < kDStrings) {
          S.key[p] = pack_key<P>(ld_pkey<P>(reinterpret_cast<const uint32_t*>(r + 1), 0));
          S.coef[p] = __hiloint2double((int)a.y, (int)a.x);
          S.act[p] = a.z;
        }
      }
      __syncthreads();
      const int n = S.n;
      // Every string reduced by its active generators, in their order: where it
      // has the pivot of one, that one is taken out.  What is left, the base,
      // names the class; what was taken out are the coordinates.
      const bool room = n <= kDStrings;
      if (room) {
        for (int i = tid; i < n; i += kDT) {
          const unsigned act = S.act[i];
          if (__popc(act) > kDRank) {  // more coordinates than a class may have
            S.bad = 1;
            continue;
          }
          DKey<P> v = S.key[i];
          unsigned f = 0, bit = 1;
          for (unsigned a = act; a; a &= a - 1, bit <<= 1) {
            const DGate<P>& G = S.gate[__ffs(a) - 1];
            uint64_t t = 0;
#pragma unroll
            for (int j = 0; j < P; ++j) t |= v.a[j] & G.pivot.a[j];
            if (t) {
#pragma unroll
              for (int j = 0; j < P; ++j) v.a[j] ^= G.p.a[j];
              f |= bit;
            }
          }
          S.coord[i] = (uint16_t)f;
          S.key[i] = v;
        }
      }
      __syncthreads();
      if (room && !S.bad) {
        for (int i = tid; i < n; i += kDT) {
          const DKey<P> v = S.key[i];
          unsigned pos = table_slot<P>(v);
          int stand = i;
          for (;;) {
            const unsigned short old = atomicCAS(&S.table[pos], (unsigned short)0, (unsigned short)(i + 1));
            if (old == 0) {
              const int c = atomicAdd(&S.classes, 1);
              S.stand[c] = (uint16_t)i;
              S.cid[i] = (uint16_t)c;
              const int rank = __popc(S.act[i]);
              if (rank) atomicAdd(&S.bin[rank], 1 << (rank - 1));
              break;
            }
            const DKey<P> w = S.key[old - 1];
            bool eq = true;
#pragma unroll
            for (int j = 0; j < P; ++j) eq &= w.a[j] == v.a[j];
            if (eq) {
              stand = old - 1;
              break;
            }
            pos = (pos + 1) & (kDTable - 1);
          }
          S.member[i] = (uint16_t)stand;
        }
      }
      __syncthreads();
      // pairs in order of falling rank: gate k of the classes concerns a prefix
      if (tid < 32) {
        const int rank = kDRank - tid;  // lane 0 the largest
        const int v = (rank >= 1) ? S.bin[rank] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
          const int y = __shfl_up_sync(kFull, x, o);
          if (lane >= o) x += y;
        }
        __syncwarp();
        if (rank >= 1) {
          S.bin[rank] = x - v;
          S.upto[rank - 1] = x;  // ranks above rank - 1
        }
      }
      __syncthreads();
      const bool laid = room && !S.bad && S.upto[0] <= kDSlots / 2;
      if (laid) {
        const int classes = S.classes;
        for (int c = tid; c < classes; c += kDT) {
          const int i = S.stand[c];
          const unsigned act = S.act[i];
          const int rank = __popc(act), size = 1 << rank;
          const int off = atomicAdd(&S.slots, size), od = rank ? atomicAdd(&S.orders, rank) : 0;
          const int pr = rank ? atomicAdd(&S.bin[rank], size / 2) : 0;
          if (off + size > kDSlots) continue;  // seen below
          DClass C;
          C.off = (uint16_t)off;
          C.pairs = (uint16_t)pr;
          C.order = (uint16_t)od;
          C.rank = (uint16_t)rank;
          S.cls[c] = C;
          const DKey<P> v = S.key[i];
          S.slot_key[off] = v;
          int k = 0;
          for (unsigned a = act; a; a &= a - 1, ++k) {
            const int g = __ffs(a) - 1;
            DKey<P> w = v;
#pragma unroll
            for (int j = 0; j < P; ++j) w.a[j] ^= S.gate[g].p.a[j];
            S.slot_key[off + (1 << k)] = w;
            S.order[od + k] = (uint8_t)g;
          }
          for (int t = 0; t < size / 2; ++t) S.pair_cls[pr + t] = (uint16_t)c;
        }
      }
      __syncthreads();
      const bool fits = laid && S.slots <= kDSlots;
      if (!fits) {  // uniform
        if (S.bad || ++s > kMaxSplit) {
          fail |= S.bad ? kPhaseRankFull : kPhaseClassFull;
          break;
        }
        continue;
      }
      const int slots = S.slots, pairs = S.upto[0];
      for (int k = tid; k < slots; k += kDT) S.slot[k] = 0.0;
      // keys of the slots with several coordinates set
      for (int t = tid; t < pairs; t += kDT) {
        const DClass C = S.cls[S.pair_cls[t]];
        const int half = 1 << (C.rank - 1), tt = t - C.pairs;
        for (int j = tt; j < 2 * half; j += half) {
          const int m = __popc(j);
          if (m < 2) continue;
          DKey<P> w;
#pragma unroll
          for (int q = 0; q < P; ++q) w.a[q] = (m & 1) ? 0ull : S.slot_key[C.off].a[q];
          for (int u = j; u; u &= u - 1) {
            const DKey<P> e = S.slot_key[C.off + (u & -u)];
#pragma unroll
            for (int q = 0; q < P; ++q) w.a[q] ^= e.a[q];
          }
          S.slot_key[C.off + j] = w;
        }
      }
      __syncthreads();
      for (int i = tid; i < n; i += kDT)
        S.slot[S.cls[S.cid[S.member[i]]].off + S.coord[i]] = S.coef[i];
      if (b % kSample == 0)
        for (int i = tid; i < n; i += kDT)
          for (unsigned a = S.act[i]; a; a &= a - 1) atomicAdd(&S.seen[__ffs(a) - 1], 1u);
      __syncthreads();
      // the k-th active gate of every class: it flips coordinate k
      for (int k = 0; k < kDRank && S.upto[k] > 0; ++k) {
        const int concerned = S.upto[k], low = (1 << k) - 1;
        for (int t = tid; t < concerned; t += kDT) {
          const DClass C = S.cls[S.pair_cls[t]];
          const DGate<P>& G = S.gate[S.order[C.order + k]];
          const int tt = t - C.pairs;
          const int j = C.off + (((tt & ~low) << 1) | (tt & low)), jr = j + (1 << k);
          const double cQ = S.slot[j], cR = S.slot[jr];
          const bool liveQ = !is_zero_bits(cQ), liveR = !is_zero_bits(cR);
          if (!liveQ && !liveR) continue;
          const DKey<P> Q = S.slot_key[j], R = S.slot_key[jr];
          const bool neg = child_negative<P>(G, Q, R);
          const double aQ = __dmul_rn(G.cth, cQ), sQ = __dmul_rn(G.sth, cQ);
          const double aR = __dmul_rn(G.cth, cR), sR = __dmul_rn(G.sth, cR);
          double nQ = __dadd_rn(aQ, with_sign(sR, !neg));
          double nR = __dadd_rn(aR, with_sign(sQ, neg));
          bool keepQ = (dbits(nQ) & kAbsMask) >= eps_bits, keepR = (dbits(nR) & kAbsMask) >= eps_bits;
          if (rule.wmax >= 0) {  // an absent member too heavy to be born stays absent
            if (!liveQ) keepQ &= __popcll(x_of<P>(Q) | z_of<P>(Q)) <= rule.wmax;
            if (!liveR) keepR &= __popcll(x_of<P>(R) | z_of<P>(R)) <= rule.wmax;
          }
          S.slot[j] = keepQ ? nQ : 0.0;
          S.slot[jr] = keepR ? nR : 0.0;
          const int was = (int)liveQ + (int)liveR, dl = (int)keepQ + (int)keepR - was;
          n_ac += was;
          upd += (long long)dl * G.after;
          skipped += (long long)dl * G.skip_after;
        }
        __syncthreads();
      }
      // survivors, listed first: the work per string is long
      uint16_t* live = reinterpret_cast<uint16_t*>(S.act);  // kDSlots entries
      for (int k0 = 0; k0 < slots; k0 += kDT) {
        const int k = k0 + tid;
        const bool keep = k < slots && !is_zero_bits(S.slot[k]);
        const unsigned bal = __ballot_sync(kFull, keep);
        unsigned p = 0;
        if (lane == 0 && bal) p = atomicAdd(&S.out_n, (unsigned)__popc(bal));
        p = __shfl_sync(kFull, p, 0) + __popc(bal & below);
        if (keep) live[p] = (uint16_t)k;
      }
      __syncthreads();
      const int n_live = (int)S.out_n;
      if (next.count) {
        for (int q = tid; q < n_live; q += kDT) {
          const int k = live[q];
          const PKey<P> K = unpack_pkey<P>(S.slot_key[k]);
          unsigned act;
          uint64_t h;
          classify<P>(K, S.next, next, act, h);
          deal<P>(out, K, S.slot[k], act, h, fail);
        }
      } else {
        if (tid == 0) S.out_base = atomicAdd(&ctl->n_next, (unsigned long long)n_live);
        __syncthreads();
        for (int q = tid; q < n_live; q += kDT) {
          const int k = live[q];
          const uint64_t at = S.out_base + (unsigned)q;
          if (at < dense.cap) {
            Key<1> K;
            K.x(0) = x_of<P>(S.slot_key[k]);
            K.z(0) = z_of<P>(S.slot_key[k]);
            st_key<1>(dense.keys, at, K);
            dense.coef[at] = S.slot[k];
            occ.add(K);
          } else {
            fail |= kPhaseTableFull;
          }
        }
      }
      while (s > 0 && ((id >> (s - 1)) & 1u)) {
        id &= ~(1u << (s - 1));
        --s;
      }
      if (s == 0) break;
      id |= 1u << (s - 1);
      if (s < s0) s = s0;
    }
  }
  if (next.count == 0) occ.flush(ctl);
  if (fail) atomicOr(&acc.st->fail, fail);
  upd = warp_sum(upd);
  skipped = warp_sum(skipped);
  n_ac = warp_sum(n_ac);
  if (lane == 0) {
    if (upd) atomicAdd(reinterpret_cast<unsigned long long*>(&acc.st->upd), (unsigned long long)upd);
    if (skipped)
      atomicAdd(reinterpret_cast<unsigned long long*>(&acc.st->skipped), (unsigned long long)skipped);
    if (n_ac) atomicAdd(&acc.st->ac, n_ac);
  }
  __syncthreads();
  if (tid < d.count) {
    if (S.seen[tid]) atomicAdd(acc.seen + d.first + tid, S.seen[tid]);
    if (blockIdx.x == 0 && !((d.skip >> tid) & 1u)) acc.touch[d.first + tid] = 1u;
  }
}

// After the last phase (one block): the statistics every path keeps, and the
// table's size.  A failed layer raises the stall flag instead, which holds off
// what is queued behind it.
__global__ void __launch_bounds__(kBlock) phase_end_kernel(DevCtl* ctl, PhaseAcc acc, unsigned n_gates) {
  __shared__ long long s_w[kBlock / 32], s_sum[4];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (acc.st->fail) {
    if (tid == 0) ctl->stall = acc.st->fail;
    return;
  }
  if (tid < 4) s_sum[tid] = 0;
  long long run = (long long)acc.st->live0, upd = 0, skipped = 0, n_skip = 0, sum_ac = 0;
  for (unsigned g0 = 0; g0 < n_gates; g0 += kBlock) {
    const unsigned g = g0 + tid;
    const bool on = g < n_gates;
    const long long d = on ? acc.delta[g] : 0;
    const unsigned long long ac = on ? acc.ac[g] : 0ull;
    const unsigned touch = on ? acc.touch[g] : 0u, seen = on ? acc.seen[g] : 0u;
    long long x = d;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(kFull, x, o);
      if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    long long before = run, all = run;
    for (int w = 0; w < kBlock / 32; ++w) {
      if (w < warp) before += s_w[w];
      all += s_w[w];
    }
    if (on) {
      const long long live = before + x - d;  // entering gate g
      upd += live;
      sum_ac += (long long)ac;
      if (!touch) {
        skipped += live;
        ++n_skip;
      }
      acc.activity[g] = live > 0 ? (float)(((double)ac + (double)kSample * seen) / (double)live) : 0.0f;
    }
    run = all;
  }
  upd = warp_sum(upd);
  skipped = warp_sum(skipped);
  n_skip = warp_sum(n_skip);
  sum_ac = warp_sum(sum_ac);
  __syncthreads();
  if (lane == 0) {
    const long long v[4] = {upd, skipped, n_skip, sum_ac};
    for (int k = 0; k < 4; ++k)
      if (v[k]) atomicAdd(reinterpret_cast<unsigned long long*>(&s_sum[k]), (unsigned long long)v[k]);
  }
  __syncthreads();
  if (tid == 0) {
    ctl->updates += (double)(s_sum[0] + acc.st->upd);
    ctl->gates_done += n_gates;
    ctl->ac_total += (unsigned long long)s_sum[3] + acc.st->ac;
    ctl->skipped_updates += (double)(s_sum[1] + acc.st->skipped);
    ctl->gates_skipped += (unsigned long long)s_sum[2];
    ctl->n_terms = ctl->n_next;
    ctl->n_live = (long long)ctl->n_next;
    ctl->after_terms = ctl->n_next;
  }
}

template <int P>
cudaError_t phase_setup() {
  static_assert(PhaseDims<P>::C < (1 << kPosBits) && 4 * PhaseDims<P>::C <= 3 * PhaseDims<P>::kSlots,
                "positions fit an index slot; an index is never full");
  static_assert(kPBlocks * (sizeof(PhaseSmem<P>) + 1024) <= 228 * 1024, "blocks per SM");
  static SmemLimit limit;
  return limit.raise(phase_kernel<P>, sizeof(PhaseSmem<P>));
}

template <int P>
cudaError_t launch_phase_pt(int warps, cudaStream_t s, const PhaseBuckets& in, const PhaseBuckets& out,
                            const PhaseDesc& d, const PhaseDesc& next,
                            const GateArgs* gates, const PhaseRule& rule, const DevTable& dense,
                            DevCtl* ctl, const PhaseAcc& acc) {
  const cudaError_t e = phase_setup<P>();
  if (e != cudaSuccess) return e;
  phase_kernel<P><<<std::max(1, warps / kPW), kPT, sizeof(PhaseSmem<P>), s>>>(
      in, out, d, next, gates, rule, dense, ctl, acc);
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_dense_p(int warps, cudaStream_t s, const PhaseBuckets& in, const PhaseBuckets& out,
                           const PhaseDesc& d, const PhaseDesc& next,
                           const GateArgs* gates, const PhaseRule& rule, const DevTable& dense,
                           DevCtl* ctl, const PhaseAcc& acc) {
  static_assert(2 * (sizeof(DenseSmem<P>) + 1024) <= 228 * 1024, "blocks per SM");
  static SmemLimit limit;
  const cudaError_t e = limit.raise(dense_phase_kernel<P>, sizeof(DenseSmem<P>));
  if (e != cudaSuccess) return e;
  // two blocks of 16 warps per SM where phase_kernel has three of 4
  const int grid = std::max(1, warps / (kPW * kPBlocks) * 2);
  dense_phase_kernel<P><<<grid, kDT, sizeof(DenseSmem<P>), s>>>(in, out, d, next, gates, rule,
                                                                dense, ctl, acc);
  return cudaGetLastError();
}

}  // namespace

int phase_words(int n) { return n <= 32 ? 1 : 2 * ((n + 63) / 64); }

int phase_warps_per_sm() { return kPW * kPBlocks; }

int phase_strings_per_warp(int P) {
  switch (P) {
    case 1: return PhaseDims<1>::C;
    case 2: return PhaseDims<2>::C;
    case 4: return PhaseDims<4>::C;
    case 6: return PhaseDims<6>::C;
    default: return PhaseDims<8>::C;
  }
}

cudaError_t launch_phase_begin(cudaStream_t s, const PhaseAcc& acc, size_t clear_bytes, DevCtl* ctl,
                               int sms) {
  const uint64_t words = clear_bytes / 4;
  const int grid = (int)std::min<uint64_t>((words + 4 * kBlock - 1) / (4 * kBlock), (uint64_t)sms * 4);
  phase_begin_kernel<<<std::max(grid, 1), kBlock, 0, s>>>(reinterpret_cast<unsigned*>(acc.st), words,
                                                          ctl);
  return cudaGetLastError();
}

#define PPP_DISPATCH(P, ...)                                \
  switch (P) {                                              \
    case 1: { constexpr int PP = 1; __VA_ARGS__; break; }   \
    case 2: { constexpr int PP = 2; __VA_ARGS__; break; }   \
    case 4: { constexpr int PP = 4; __VA_ARGS__; break; }   \
    case 6: { constexpr int PP = 6; __VA_ARGS__; break; }   \
    case 8: { constexpr int PP = 8; __VA_ARGS__; break; }   \
    default: return cudaErrorInvalidValue;                  \
  }

cudaError_t launch_phase_deal(int P, int grid, cudaStream_t s, const DevTable& src, uint64_t T,
                              int use_eps, const PhaseBuckets& out, const PhaseDesc& d,
                              const GateArgs* gates, const PhaseAcc& acc) {
  PPP_DISPATCH(P, (phase_deal_kernel<PP><<<grid, kBlock, 0, s>>>(src.keys, src.coef, T, use_eps, out, d,
                                                                 gates, acc)));
  return cudaGetLastError();
}

cudaError_t launch_phase(int P, int warps, cudaStream_t s, const PhaseBuckets& in,
                         const PhaseBuckets& out, const PhaseDesc& d,
                         const PhaseDesc& next, const GateArgs* gates, const PhaseRule& rule,
                         const DevTable& dense, DevCtl* ctl, const PhaseAcc& acc) {
  if (d.dense && P <= 2) {
    if (P == 1) return launch_dense_p<1>(warps, s, in, out, d, next, gates, rule, dense, ctl, acc);
    return launch_dense_p<2>(warps, s, in, out, d, next, gates, rule, dense, ctl, acc);
  }
  PPP_DISPATCH(P, return (launch_phase_pt<PP>(warps, s, in, out, d, next, gates, rule, dense,
                                              ctl, acc)));
  return cudaErrorInvalidValue;
}

cudaError_t launch_phase_end(cudaStream_t s, DevCtl* ctl, const PhaseAcc& acc, unsigned n_gates) {
  phase_end_kernel<<<1, kBlock, 0, s>>>(ctl, acc, n_gates);
  return cudaGetLastError();
}

}  // namespace ppk
