// Merge by buckets: the merge loop of Algorithms 2 and 3 without a hash index in
// global memory.
//
// Every string is mapped to its representative and dealt into a bucket by the
// representative's hash, so equal ones meet in one bucket; a block takes a bucket
// into shared memory, adds equal strings up there and appends what truncation
// keeps to the destination.  Two passes over the table, one of them scattered, a
// sector a string, in the place of one with three random sectors and an atomic
// per string, and no index to clear (8 to 16 bytes per entry of capacity).
// 1.95 million strings of 32 sites into 975 thousand under Z_n: 65 us dealt (82
// with key, coefficient and hash in arrays of their own) and 44 us merged, where
// the index took 0.35 ms with its clearing.  Bound by the atomics and scattered
// sectors of the deal, and by the probes in shared memory after it.
//
// A bucket larger than a block's room is done in parts, split by further bits of
// the hash.  A full bucket, or more equal strings than a block holds, raises
// kMergeFull; the source is never written, and the caller merges it by the hash
// index.
#include <algorithm>

#include "pp_phase.cuh"
#include "pp_smem_limit.h"

namespace ppk {
namespace {

constexpr int kMT = 256;

template <int P>
struct MergeSmem {
  static constexpr int C = P <= 4 ? 1024 : 512;
  PKey<P> key[C];
  double coef[C], sum[C];
  uint16_t table[2 * C];
  int n;
  unsigned out_n;
  unsigned long long out_base;
};

// A string in its bucket: key words and coefficient in units of 16 bytes, so that
// it is scattered in the fewest sectors (one of 32 bytes up to 64 sites).
template <int P>
__device__ __forceinline__ void st_rec(ulonglong2* to, uint64_t i, const PKey<P>& k, double c) {
  constexpr int U = (P + 2) / 2;
  uint64_t r[2 * U];
  r[2 * U - 1] = 0ull;
#pragma unroll
  for (int j = 0; j < P; ++j) r[j] = (uint64_t)k.w[2 * j] | ((uint64_t)k.w[2 * j + 1] << 32);
  r[P] = (uint64_t)__double_as_longlong(c);
#pragma unroll
  for (int j = 0; j < U; ++j) to[i * U + j] = make_ulonglong2(r[2 * j], r[2 * j + 1]);
}

template <int P>
__device__ __forceinline__ double ld_rec(const ulonglong2* from, uint64_t i, PKey<P>& k) {
  constexpr int U = (P + 2) / 2;
  uint64_t r[2 * U];
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const ulonglong2 v = from[i * U + j];
    r[2 * j] = v.x;
    r[2 * j + 1] = v.y;
  }
#pragma unroll
  for (int j = 0; j < P; ++j) {
    k.w[2 * j] = (uint32_t)r[j];
    k.w[2 * j + 1] = (uint32_t)(r[j] >> 32);
  }
  return __longlong_as_double((long long)r[P]);
}

__device__ __forceinline__ bool merge_off(const DevCtl* ctl, const unsigned* fail, int guarded) {
  return (guarded && queued_layer_stopped(ctl)) || *reinterpret_cast<const volatile unsigned*>(fail) != 0u;
}

// Counters and the append cursor; a layer that stopped keeps its own.
__global__ void __launch_bounds__(kBlock)
    merge_begin_kernel(unsigned* words, uint64_t n, DevCtl* ctl, int guarded) {
  if (guarded && queued_layer_stopped(ctl)) n = 1;  // the flag alone
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) words[i] = 0u;
  if (blockIdx.x == 0 && threadIdx.x == 0 && n > 1) {
    ctl->n_next = 0;
    for (int j = 0; j < 2 * kMaxW; ++j) ctl->occ[j] = 0ull;
  }
}

template <int P, int G>
__global__ void __launch_bounds__(kBlock)
    merge_deal_kernel(const uint64_t* __restrict__ keys, const double* __restrict__ coef,
                      uint64_t count, const unsigned long long* count_dev, int skip_zero, int n, int lx,
                      MergeBuckets out, const DevCtl* ctl,
                      int guarded) {
  constexpr int W = (P + 1) / 2;
  if (merge_off(ctl, out.fail, guarded)) return;
  const uint64_t T = count_dev ? *count_dev : count;
  unsigned bad = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < T; i += stride) {
    const double c = coef[i];
    if (skip_zero && c == 0.0) continue;
    Key<W> K = ld_key<W>(keys, i);
    canon<W, G>(K, n, lx);
    PKey<P> k;
#pragma unroll
    for (int j = 0; j < P; ++j) {
      k.w[j] = (uint32_t)(K.x(j / 2) >> (32 * (j & 1)));
      k.w[P + j] = (uint32_t)(K.z(j / 2) >> (32 * (j & 1)));
    }
    const unsigned b = (unsigned)(((string_hash<P>(k, 0u) >> 32) * (uint64_t)out.nb) >> 32);
    const unsigned p = atomicAdd(out.cnt + b, 1u);
    if (p < out.cg)
      st_rec<P>(out.rec, (uint64_t)b * out.cg + p, k, c);
    else
      bad = 1;
  }
  if (bad) atomicOr(out.fail, kMergeFull);
}

template <int P>
__global__ void __launch_bounds__(kMT)
    merge_bucket_kernel(MergeBuckets in, double eps, DevTable dst, DevCtl* ctl, int guarded) {
  extern __shared__ __align__(16) unsigned char merge_raw[];
  MergeSmem<P>& S = *reinterpret_cast<MergeSmem<P>*>(merge_raw);
  constexpr int C = MergeSmem<P>::C, W = (P + 1) / 2;
  if (__syncthreads_or(merge_off(ctl, in.fail, guarded))) return;  // the whole block or none of it
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned below = (1u << lane) - 1u;
  unsigned bad = 0;
  OccAcc<W> occ;
  for (unsigned b = blockIdx.x; b < in.nb; b += gridDim.x) {
    const int cnt = (int)min(in.cnt[b], in.cg);
    if (cnt == 0) continue;
    const uint64_t base = (uint64_t)b * in.cg;
    int s0 = 0;  // parts, as in phase_kernel
    while ((cnt >> s0) > C * 7 / 8) ++s0;
    int s = s0;
    unsigned id = 0;
    for (;;) {
      __syncthreads();
      for (int k = tid; k < C; k += kMT) reinterpret_cast<unsigned*>(S.table)[k] = 0u;
      if (tid == 0) {
        S.n = 0;
        S.out_n = 0;
      }
      __syncthreads();
      for (int i0 = 0; i0 < cnt; i0 += kMT) {
        const int i = i0 + tid;
        PKey<P> K;
        double c = 0.0;
        bool mine = i < cnt;
        if (mine) {
          c = ld_rec<P>(in.rec, base + i, K);
          if (s > 0) mine = ((unsigned)string_hash<P>(K, 0u) & ((1u << s) - 1u)) == id;
        }
        const unsigned bal = __ballot_sync(kFull, mine);
        int p = 0;
        if (lane == 0 && bal) p = atomicAdd(&S.n, __popc(bal));
        p = __shfl_sync(kFull, p, 0) + __popc(bal & below);
        if (mine && p < C) {
          S.key[p] = K;
          S.coef[p] = S.sum[p] = c;
        }
      }
      __syncthreads();
      const int n = S.n;
      if (n > C) {  // uniform
        if (++s > kMaxSplit) {
          bad |= kMergeFull;
          break;
        }
        continue;
      }
      // one of equal strings stands for them, the others add to its sum
      for (int i = tid; i < n; i += kMT) {
        const PKey<P> K = S.key[i];
        unsigned pos = (unsigned)(string_hash<P>(K, 0x2545F491u) >> 32) & (2 * C - 1);
        for (;;) {
          const unsigned short old = atomicCAS(&S.table[pos], (unsigned short)0, (unsigned short)(i + 1));
          if (old == 0) break;
          const PKey<P> Q = S.key[old - 1];
          bool eq = true;
#pragma unroll
          for (int j = 0; j < 2 * P; ++j) eq &= Q.w[j] == K.w[j];
          if (eq) {
            atomicAdd(&S.sum[old - 1], S.coef[i]);
            break;
          }
          pos = (pos + 1) & (2 * C - 1);
        }
      }
      __syncthreads();
      for (int pass = 0; pass < 2; ++pass) {  // count, reserve, then write
        for (int i0 = 0; i0 < 2 * C; i0 += kMT) {
          const int e = S.table[i0 + tid];
          const double c = e ? S.sum[e - 1] : 0.0;
          const bool keep = e && (eps > 0.0 ? fabs(c) >= eps : true);
          const unsigned bal = __ballot_sync(kFull, keep);
          unsigned p = 0;
          if (lane == 0 && bal) p = atomicAdd(&S.out_n, (unsigned)__popc(bal));
          p = __shfl_sync(kFull, p, 0) + __popc(bal & below);
          if (pass == 1 && keep) {
            const uint64_t at = S.out_base + p;
            if (at < dst.cap) {
              const Key<W> K = table_key<P>(S.key[e - 1]);
              st_key<W>(dst.keys, at, K);
              dst.coef[at] = c;
              occ.add(K);
            } else {
              bad |= kMergeFull;
            }
          }
        }
        __syncthreads();
        if (pass == 0) {
          if (tid == 0) {
            S.out_base = atomicAdd(&ctl->n_next, (unsigned long long)S.out_n);
            S.out_n = 0;
          }
          __syncthreads();
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
  occ.flush(ctl);
  if (bad) atomicOr(in.fail, bad);
}

// The merged table's size, or the failure in the stall flag.
__global__ void merge_end_kernel(const unsigned* fail, DevCtl* ctl, int guarded) {
  if (guarded && queued_layer_stopped(ctl)) return;
  if (*fail) {
    ctl->stall = kMergeFull;
    return;
  }
  ctl->n_terms = ctl->n_next;
  ctl->n_live = (long long)ctl->n_next;
}

template <int P, int G>
cudaError_t merge_pg(const MergeBuckets& m, cudaStream_t s, const DevTable& src, uint64_t count,
                     const unsigned long long* count_dev, int skip_zero, int n, int lx, double eps,
                     const DevTable& dst, DevCtl* ctl, int sms, int guarded) {
  const uint64_t words = 64 + m.nb;
  merge_begin_kernel<<<(int)std::min<uint64_t>((words + 1023) / 1024, (uint64_t)sms * 4), kBlock, 0, s>>>(
      m.fail, words, ctl, guarded);
  const uint64_t bound = count_dev ? src.cap : count;
  merge_deal_kernel<P, G><<<(int)std::max<uint64_t>(1, std::min<uint64_t>((bound + kBlock - 1) / kBlock,
                                                                          (uint64_t)sms * 8)),
                            kBlock, 0, s>>>(src.keys, src.coef, count, count_dev, skip_zero, n, lx,
                                            m, ctl, guarded);
  static SmemLimit limit;
  const cudaError_t e = limit.raise(merge_bucket_kernel<P>, sizeof(MergeSmem<P>));
  if (e != cudaSuccess) return e;
  const int per_sm = std::min<int>(8, (int)(226 * 1024 / (sizeof(MergeSmem<P>) + 1024)));
  merge_bucket_kernel<P><<<(int)std::min<uint64_t>(m.nb, (uint64_t)sms * per_sm), kMT,
                           sizeof(MergeSmem<P>), s>>>(m, eps, dst, ctl, guarded);
  merge_end_kernel<<<1, 1, 0, s>>>(m.fail, ctl, guarded);
  return cudaGetLastError();
}

size_t al256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

// Buckets of 600 strings on average (a block's room is 1024), room for twice that
// and four orbits of all 2 n members: hashes spread evenly over the orbits.
MergeBuckets merge_buckets(int n, uint64_t count, int sms) {
  MergeBuckets m;
  const int P = phase_words(n);
  m.nb = (unsigned)std::max<uint64_t>((uint64_t)sms * 2, (count + 599) / 600);
  m.cg = (unsigned)((2 * count / m.nb + 8 * (uint64_t)n + 256) / 8 * 8);
  m.bytes = al256((64 + (size_t)m.nb) * 4) + al256((size_t)m.nb * m.cg * ((P + 2) / 2) * 16);
  m.fail = m.cnt = nullptr;
  m.rec = nullptr;
  return m;
}

void place_merge_buckets(MergeBuckets& m, void* scratch) {
  m.fail = static_cast<unsigned*>(scratch);
  m.cnt = m.fail + 64;
  m.rec = reinterpret_cast<ulonglong2*>(static_cast<unsigned char*>(scratch) +
                                        al256((64 + (size_t)m.nb) * 4));
}

cudaError_t launch_merge_buckets(const MergeBuckets& m, int n, int group, cudaStream_t s,
                                 const DevTable& src, uint64_t count,
                                 const unsigned long long* count_dev, int skip_zero, double eps,
                                 const DevTable& dst, DevCtl* ctl, int sms, int guarded) {
  const int lx = group >> 8;
#define PPM_P(GG)                                                                                     \
  switch (phase_words(n)) {                                                                           \
    case 1: return merge_pg<1, GG>(m, s, src, count, count_dev, skip_zero, n, lx, eps, dst, ctl, sms, guarded); \
    case 2: return merge_pg<2, GG>(m, s, src, count, count_dev, skip_zero, n, lx, eps, dst, ctl, sms, guarded); \
    case 4: return merge_pg<4, GG>(m, s, src, count, count_dev, skip_zero, n, lx, eps, dst, ctl, sms, guarded); \
    case 6: return merge_pg<6, GG>(m, s, src, count, count_dev, skip_zero, n, lx, eps, dst, ctl, sms, guarded); \
    case 8: return merge_pg<8, GG>(m, s, src, count, count_dev, skip_zero, n, lx, eps, dst, ctl, sms, guarded); \
    default: return cudaErrorInvalidValue;                                                            \
  }
  switch (group & 0xFF) {
    case 0: PPM_P(0);
    case 1: PPM_P(1);
    case 3: PPM_P(3);
    case 4: PPM_P(4);
    default: return cudaErrorInvalidValue;
  }
#undef PPM_P
}

}  // namespace ppk
