// Phases (pp_phase.cu) of batched layers: every string carries a row of B
// coefficients, FP64 or FP32.
//
// Strings travel through the buckets with the number of their row; a block takes
// a bucket, finds its classes, and for one class after the other lays the rows of
// its members out as a dense array [2^r][B] in shared memory (in global memory
// beyond what that holds).  Columns are independent but for the rule that a row
// is kept while some column is large, so a thread owns a column through all the
// class's gates, and the block meets twice per gate to exchange which rows live.
// Surviving rows are written once, behind one another, into the rows of the next
// phase.
//
// Why: one pass per gate read and wrote a row of every pair from L2 or HBM at
// every gate, after a grid barrier and a lookup per string (17 us a gate at 10^3
// to 10^4 strings of 256 FP64 columns).  Here a row moves twice per phase of up
// to 32 gates, and the products and sums of the pairs are what is left.
#include <algorithm>

#include "pp_phase.cuh"
#include "pp_smem_limit.h"

namespace ppk {
namespace {

constexpr int kRStrings = 256;         // strings of a part
constexpr int kRTable = 512;           // hash slots of the class lookup
constexpr int kRMembers = 1 << kDRank; // rows of a class at most

__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rflip(float v, bool neg) {
  return __int_as_float(__float_as_int(v) ^ (neg ? (int)0x80000000u : 0));
}
__device__ __forceinline__ double rflip(double v, bool neg) { return with_sign(v, neg); }
// |v| >= eps on bit patterns, in the storage type
__device__ __forceinline__ bool rbig(float v, uint64_t eb) {
  return (__float_as_uint(v) & 0x7FFFFFFFu) >= (uint32_t)eb;
}
__device__ __forceinline__ bool rbig(double v, uint64_t eb) { return (dbits(v) & kAbsMask) >= eb; }

template <typename T>
__device__ __forceinline__ uint64_t row_eps_bits(double eps) {
  if (sizeof(T) == 4) return (uint64_t)__float_as_uint((float)eps);
  return dbits(eps);
}

template <int P>
struct RowsSmem {
  DGate<P> gate[kPhaseGates];
  NextGens<P> mine, next;
  DKey<P> key[kRStrings];        // string, then the base of its class
  DKey<P> member_key[kRMembers]; // of the class in hand
  uint32_t act[kRStrings], row[kRStrings];
  uint32_t alive[2][kRMembers / 32];
  uint16_t coord[kRStrings], member[kRStrings], stand[kRStrings];
  uint16_t table[kRTable];
  uint16_t first[kRStrings + 1];  // members of class c: list[first[c], first[c + 1])
  uint16_t list[kRStrings];
  uint16_t count[kRStrings];
  uint16_t cls[kRStrings];        // class of a standing string
  int n, classes, bad;
  unsigned long long out_base;
  unsigned seen[kPhaseGates];
};

// Live rows of a dense table into the buckets of the first phase; the row number
// travels in the place of the coefficient.
template <int P>
__global__ void __launch_bounds__(kBlock)
    rows_deal_kernel(const uint64_t* __restrict__ keys, const unsigned char* __restrict__ alive,
                     uint64_t T, PhaseBuckets out, PhaseDesc d,
                     const GateArgs* __restrict__ gates, PhaseAcc acc) {
  __shared__ __align__(16) NextGens<P> next;
  __shared__ unsigned s_live;
  if (threadIdx.x == 0) s_live = 0;
  load_generators<P>(next, gates, d);
  unsigned fail = 0, live = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < T; i += stride) {
    if (!alive[i]) continue;
    const PKey<P> K = ld_table_key<P>(keys, i);
    ++live;
    unsigned act;
    uint64_t h;
    classify<P>(K, next, d, act, h);
    deal<P>(out, K, __longlong_as_double((long long)i), act, h, fail);
  }
  live = __reduce_add_sync(kFull, live);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_live, live);
  if (fail) atomicOr(&acc.st->fail, fail);
  __syncthreads();
  if (threadIdx.x == 0 && s_live) atomicAdd(&acc.st->live0, (unsigned long long)s_live);
}

// One phase.  src / dst: rows of B columns; dst_cap rows.  smem_rows: rows of a
// class that fit in shared memory behind RowsSmem; spill: kRMembers rows per
// block for larger ones.  n_out counts the rows written to dst.  With
// next.count == 0 the keys and liveness of `dense` are written too.
template <int P, typename T>
__global__ void __launch_bounds__(256)
    rows_phase_kernel(PhaseBuckets in, PhaseBuckets out, PhaseDesc d,
                      PhaseDesc next, const GateArgs* __restrict__ gates, const T* __restrict__ src,
                      T* dst, uint64_t dst_cap, unsigned long long* n_out, int B, int use_eps,
                      double eps, int wmax, int smem_rows, T* spill, DevTable dense, DevCtl* ctl,
                      PhaseAcc acc) {
  extern __shared__ __align__(16) unsigned char phase_raw[];
  RowsSmem<P>& S = *reinterpret_cast<RowsSmem<P>*>(phase_raw);
  T* const shared_rows = reinterpret_cast<T*>(phase_raw + (sizeof(RowsSmem<P>) + 15) / 16 * 16);
  T* const spill_rows = spill + (uint64_t)blockIdx.x * kRMembers * B;
  if (__syncthreads_or(*reinterpret_cast<const volatile unsigned*>(&acc.st->fail) != 0u)) return;
  const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31;
  const uint64_t eb = use_eps ? row_eps_bits<T>(eps) : 0ull;
  load_generators<P>(S.mine, gates, d);
  load_generators<P>(S.next, gates, next);
  for (int g = tid; g < d.count; g += NT) {
    const GateArgs& a = gates[d.first + g];
    DGate<P>& G = S.gate[g];
    G.p = pack_key<P>(S.mine.gen[g]);
    G.pivot = pack_key<P>(S.mine.pivot[g]);
    G.pyy = a.pyy;
    G.after = d.after + d.count - 1 - g;
    G.skip_after = d.skip_after + (g + 1 < 32 ? __popc(d.skip >> (g + 1)) : 0);
  }
  for (int g = tid; g < kPhaseGates; g += NT) S.seen[g] = 0;
  unsigned fail = 0;
  long long upd = 0, skipped = 0;  // of thread 0
  unsigned long long n_ac = 0;
  OccAcc<1> occ;
  for (unsigned b = blockIdx.x; b < in.nb; b += gridDim.x) {
    const int cnt = (int)min(in.cnt[b], in.cg);
    if (cnt == 0) continue;
    const uint64_t base = (uint64_t)b * in.cg;
    int s0 = 0;
    while ((cnt >> s0) > kRStrings * 3 / 4) ++s0;
    int s = s0;
    unsigned id = 0;
    for (;;) {
      __syncthreads();  // the last part's readers are done
      for (int k = tid; k < kRTable; k += NT) S.table[k] = 0;
      for (int k = tid; k < kRStrings; k += NT) S.count[k] = 0;
      if (tid == 0) S.n = S.classes = S.bad = 0;
      __syncthreads();
      for (int i = tid; i < cnt; i += NT) {
        const uint4* r = in.rec + (base + i) * kRecord<P>;
        const uint4 head = r[0];
        const uint2 m = make_uint2(head.z, head.w);
        if ((m.y & ((1u << s) - 1u)) != id) continue;
        const int p = atomicAdd(&S.n, 1);
        if (p >= kRStrings) continue;
        S.row[p] = head.x;
        S.act[p] = m.x;
        DKey<P> v = pack_key<P>(ld_pkey<P>(reinterpret_cast<const uint32_t*>(r + 1), 0));
        unsigned f = 0;
        if (__popc(m.x) > kDRank) {
          S.bad = 1;
        } else {  // as in dense_phase_kernel: the base and the coordinates
          unsigned bit = 1;
          for (unsigned a = m.x; a; a &= a - 1, bit <<= 1) {
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
        }
        S.key[p] = v;
        S.coord[p] = (uint16_t)f;
      }
      __syncthreads();
      const int n = S.n;
      const bool fits = n <= kRStrings && !S.bad;
      if (!fits) {  // uniform
        if (S.bad || ++s > kMaxSplit) {
          fail |= S.bad ? kPhaseRankFull : kPhaseClassFull;
          break;
        }
        continue;
      }
      for (int i = tid; i < n; i += NT) {
        const DKey<P> v = S.key[i];
        unsigned pos = table_slot<P>(v) & (kRTable - 1);
        int stand = i;
        for (;;) {
          const unsigned short old = atomicCAS(&S.table[pos], (unsigned short)0, (unsigned short)(i + 1));
          if (old == 0) {
            const int c = atomicAdd(&S.classes, 1);
            S.stand[c] = (uint16_t)i;
            S.cls[i] = (uint16_t)c;
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
          pos = (pos + 1) & (kRTable - 1);
        }
        S.member[i] = (uint16_t)stand;
        if (b % kSample == 0)
          for (unsigned a = S.act[i]; a; a &= a - 1) atomicAdd(&S.seen[__ffs(a) - 1], 1u);
      }
      __syncthreads();
      const int classes = S.classes;
      if (tid == 0) {  // members listed class by class (n <= 256)
        for (int i = 0; i < n; ++i) S.count[S.cls[S.member[i]]]++;
        int at = 0;
        for (int c = 0; c < classes; ++c) {
          S.first[c] = (uint16_t)at;
          at += S.count[c];
          S.count[c] = S.first[c];
        }
        S.first[classes] = (uint16_t)at;
        for (int i = 0; i < n; ++i) S.list[S.count[S.cls[S.member[i]]]++] = (uint16_t)i;
      }
      __syncthreads();
      for (int c = 0; c < classes; ++c) {
        const int head = S.stand[c], m0 = S.first[c], m1 = S.first[c + 1];
        const unsigned act = S.act[head];
        const int rank = __popc(act), size = 1 << rank, words = (size + 31) / 32;
        T* const D = size <= smem_rows ? shared_rows : spill_rows;
        for (int j = tid; j < size; j += NT) {
          DKey<P> w = S.key[head];
          int k = 0;
          for (unsigned a = act; a; a &= a - 1, ++k)
            if ((j >> k) & 1) {
              const DKey<P> g = S.gate[__ffs(a) - 1].p;
#pragma unroll
              for (int q = 0; q < P; ++q) w.a[q] ^= g.a[q];
            }
          S.member_key[j] = w;
        }
        for (int w = tid; w < words; w += NT) S.alive[0][w] = 0u;
        __syncthreads();
        for (int m = m0 + tid; m < m1; m += NT) {
          const int j = S.coord[S.list[m]];
          atomicOr(&S.alive[0][j >> 5], 1u << (j & 31));
        }
        for (int m = m0; m < m1; ++m) {
          const int i = S.list[m];
          const T* r = src + (uint64_t)S.row[i] * B;
          T* to = D + (uint64_t)S.coord[i] * B;
          for (int col = tid; col < B; col += NT) to[col] = r[col];
        }
        __syncthreads();
        int cur = 0, live = m1 - m0;
        unsigned a = act;
        for (int k = 0; k < rank; ++k, a &= a - 1) {
          const int g = __ffs(a) - 1;
          const DGate<P>& G = S.gate[g];
          const T* cs = static_cast<const T*>(gates[d.first + g].csb);
          const uint32_t* al = S.alive[cur];
          uint32_t* nx = S.alive[cur ^ 1];
          for (int w = tid; w < words; w += NT) nx[w] = 0u;
          __syncthreads();
          for (int c0 = 0; c0 < B; c0 += NT) {
            const int col = c0 + tid;
            const bool on = col < B;
            const T cv = on ? cs[col] : (T)0, sv = on ? cs[B + col] : (T)0;
            for (int t = 0; t < size / 2; ++t) {
              const int low = (1 << k) - 1, j = ((t & ~low) << 1) | (t & low), jr = j + (1 << k);
              const bool lQ = (al[j >> 5] >> (j & 31)) & 1u, lR = (al[jr >> 5] >> (jr & 31)) & 1u;
              if (!lQ && !lR) continue;  // uniform
              const DKey<P> Q = S.member_key[j], R = S.member_key[jr];
              const bool ng = child_negative<P>(G, Q, R);
              bool mayQ = true, mayR = true;  // an absent member too heavy to be born stays absent
              if (wmax >= 0) {
                if (!lQ) mayQ = __popcll(x_of<P>(Q) | z_of<P>(Q)) <= wmax;
                if (!lR) mayR = __popcll(x_of<P>(R) | z_of<P>(R)) <= wmax;
              }
              bool bigQ = false, bigR = false;
              if (on) {
                const T dq = lQ ? D[(uint64_t)j * B + col] : (T)0, dr = lR ? D[(uint64_t)jr * B + col] : (T)0;
                const T sQ = rmul(sv, dq), sR = rmul(sv, dr);
                const T nq = radd(rmul(cv, dq), rflip(sR, !ng));
                const T nr = radd(rmul(cv, dr), rflip(sQ, ng));
                D[(uint64_t)j * B + col] = nq;
                D[(uint64_t)jr * B + col] = nr;
                bigQ = !use_eps || rbig(nq, eb);
                bigR = !use_eps || rbig(nr, eb);
              }
              bigQ = __any_sync(kFull, bigQ) && mayQ;
              bigR = __any_sync(kFull, bigR) && mayR;
              if (lane == 0) {
                if (bigQ) atomicOr(&nx[j >> 5], 1u << (j & 31));
                if (bigR) atomicOr(&nx[jr >> 5], 1u << (jr & 31));
              }
            }
          }
          __syncthreads();
          cur ^= 1;
          if (tid == 0) {
            int now = 0;
            for (int w = 0; w < words; ++w) now += __popc(S.alive[cur][w]);
            n_ac += (unsigned long long)live;
            upd += (long long)(now - live) * G.after;
            skipped += (long long)(now - live) * G.skip_after;
            live = now;
          }
        }
        if (tid == 0 && live) S.out_base = atomicAdd(n_out, (unsigned long long)live);
        __syncthreads();
        const uint32_t* al = S.alive[cur];
        int rows = 0;
        for (int w = 0; w < words; ++w) rows += __popc(al[w]);
        if (rows && S.out_base + (uint64_t)rows > dst_cap) {
          fail |= kPhaseTableFull;
        } else if (rows) {
          const uint64_t ob = S.out_base;
          for (int j = tid; j < size; j += NT) {
            if (!((al[j >> 5] >> (j & 31)) & 1u)) continue;
            uint64_t at = ob + (unsigned)__popc(al[j >> 5] & ((1u << (j & 31)) - 1u));
            for (int w = 0; w < (j >> 5); ++w) at += (unsigned)__popc(al[w]);
            const DKey<P> w = S.member_key[j];
            if (next.count) {
              const PKey<P> K = unpack_pkey<P>(w);
              unsigned na;
              uint64_t h;
              classify<P>(K, S.next, next, na, h);
              deal<P>(out, K, __longlong_as_double((long long)at), na, h, fail);
            } else {
              Key<1> K;
              K.x(0) = x_of<P>(w);
              K.z(0) = z_of<P>(w);
              st_key<1>(dense.keys, at, K);
              dense.alive[at] = 1;
              occ.add(K);
            }
          }
          uint64_t at = ob;
          for (int j = 0; j < size; ++j) {
            if (!((al[j >> 5] >> (j & 31)) & 1u)) continue;
            const T* r = D + (uint64_t)j * B;
            T* to = dst + at * B;
            for (int col = tid; col < B; col += NT) to[col] = r[col];
            ++at;
          }
        }
        __syncthreads();  // the class's arrays are laid out anew
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
  if (tid == 0) {
    if (upd) atomicAdd(reinterpret_cast<unsigned long long*>(&acc.st->upd), (unsigned long long)upd);
    if (skipped)
      atomicAdd(reinterpret_cast<unsigned long long*>(&acc.st->skipped), (unsigned long long)skipped);
    if (n_ac) atomicAdd(&acc.st->ac, n_ac);
  }
  __syncthreads();
  for (int g = tid; g < d.count; g += NT) {
    if (S.seen[g]) atomicAdd(acc.seen + d.first + g, S.seen[g]);
    if (blockIdx.x == 0 && !((d.skip >> g) & 1u)) acc.touch[d.first + g] = 1u;
  }
}

template <int P, typename T>
cudaError_t launch_rows_pt(const RowsLaunch& L, cudaStream_t s, const PhaseBuckets& in,
                           const PhaseBuckets& out, const PhaseDesc& d,
                           const PhaseDesc& next, const GateArgs* gates, const PhaseRule& rule,
                           const void* src, void* dst, uint64_t dst_cap, unsigned long long* n_out,
                           void* spill, const DevTable& dense, DevCtl* ctl, const PhaseAcc& acc) {
  static SmemLimit limit;
  const cudaError_t e = limit.raise(rows_phase_kernel<P, T>, 227 * 1024);
  if (e != cudaSuccess) return e;
  rows_phase_kernel<P, T><<<L.grid, L.threads, L.smem, s>>>(
      in, out, d, next, gates, static_cast<const T*>(src), static_cast<T*>(dst), dst_cap, n_out,
      dense.B, rule.use_eps, rule.eps, rule.wmax, L.smem_rows, static_cast<T*>(spill), dense, ctl, acc);
  return cudaGetLastError();
}

}  // namespace

RowsLaunch rows_launch(int P, int B, int esize, int sms) {
  RowsLaunch L;
  L.threads = std::min(256, std::max(64, (B + 31) / 32 * 32));
  const size_t fixed = ((P == 1 ? sizeof(RowsSmem<1>) : sizeof(RowsSmem<2>)) + 15) / 16 * 16;
  // two blocks per SM where that leaves 8 rows, all of them one block otherwise
  const size_t row = (size_t)B * esize, two = 112 * 1024;
  const size_t room = fixed + 8 * row <= two ? two : 226 * 1024;
  L.smem_rows = (int)std::min<size_t>(kRMembers, (room - fixed) / row);
  L.smem = fixed + (size_t)L.smem_rows * row;
  const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(8, 226 * 1024 / (L.smem + 1024)));
  L.grid = sms * per_sm;
  L.spill_rows = (size_t)L.grid * kRMembers;
  return L;
}

cudaError_t launch_rows_deal(int P, int grid, cudaStream_t s, const DevTable& src, uint64_t T,
                             const PhaseBuckets& out, const PhaseDesc& d,
                             const GateArgs* gates, const PhaseAcc& acc) {
  if (P == 1)
    rows_deal_kernel<1><<<grid, kBlock, 0, s>>>(src.keys, src.alive, T, out, d, gates, acc);
  else
    rows_deal_kernel<2><<<grid, kBlock, 0, s>>>(src.keys, src.alive, T, out, d, gates, acc);
  return cudaGetLastError();
}

cudaError_t launch_rows_phase(int P, const RowsLaunch& L, cudaStream_t s, const PhaseBuckets& in,
                              const PhaseBuckets& out, const PhaseDesc& d,
                              const PhaseDesc& next, const GateArgs* gates, const PhaseRule& rule,
                              const void* src, void* dst, uint64_t dst_cap, unsigned long long* n_out,
                              void* spill, const DevTable& dense, DevCtl* ctl, const PhaseAcc& acc) {
#define PPR(PP, TT)                                                                                \
  return launch_rows_pt<PP, TT>(L, s, in, out, d, next, gates, rule, src, dst, dst_cap, n_out, \
                                spill, dense, ctl, acc)
  if (P == 1) {
    if (dense.f32) PPR(1, float);
    PPR(1, double);
  }
  if (dense.f32) PPR(2, float);
  PPR(2, double);
#undef PPR
}

}  // namespace ppk
