// Role-conditional allocation and per-bucket top-k (Section 4.1, Algorithm 1):
// pool the scores (optional), count the roles, split the budget ceil(B n)
// across role buckets, and keep the top-q_r tokens of every bucket, ties to the
// lower index.  A cluster of C CTAs per (layer, sequence, KV head), C = 1 to 8,
// holds the unit's keys in shared memory, each CTA a contiguous slice;
// everything after the fp32 -> ordered-key mapping is integer, so the kept set
// is bit-exact for a given score row and does not depend on C.
//
// Slots.  Shared memory holds the unit in "slots": slot s is token s - off,
// where off = (start address of the score row / 4) mod 4, so that every group
// of four slots is one aligned 16-byte vector both in global and in shared
// memory.  Slots outside [off, off + n) have role 0xFF and are never kept.
// Rank k of the cluster owns groups [k gs, (k + 1) gs).
//
// The threshold of each bucket is found by a radix descent over the keys'
// bits, most significant first:
//   pass 1  load, pool, key; per role, a histogram of the key's bits
//           30..31-NB (the top bit is shared by every key when all scores
//           have one sign): exponent and leading mantissa bits; role counts.
//           Under GLOBAL there is one bucket, so one histogram of every
//           eligible token.
//   quotas  one warp, lane r for role r (water-filling, largest remainders),
//           from the ranks' counts, in every rank alike.
//   first digit from the ranks' pass-1 histograms, bucket b by rank b mod C;
//           while the keys at the threshold digits would overflow the list, a
//           full pass over the slots per 8 more bits.
//   pass 2  every token is decided (kept / dropped) unless its key prefix is
//           its bucket's threshold prefix; those "candidates" (a few
//           percent) go to the rank's list in shared memory.
//   list    the remaining bits in 8-bit rounds over the lists, every rank
//           reading the ranks' digit counts; ties at the threshold are ranked
//           in index order; the kept ones join the bits.
// A unit with a NaN, keys of both signs, or more candidates than a list
// holds 4 to 5 bits above the bottom takes the general path: four 8-bit
// rounds over all slots.
// Kept positions are then written in ascending order from a scan of the bit
// words, each rank at the offset of the ranks before it.
//
// Rows longer than kSmemMaxN tokens in batches of more units than a few waves
// of clusters (streaming mode, one CTA per unit) do not keep their keys:
// every pass recomputes a group's pooled keys from the score row (read again
// from L2), the first-digit histograms count in 32 bits and a candidate-list
// entry carries its key beside (bucket << 24) | slot.
//
// The ranks read each other's counts and histograms through distributed
// shared memory, one cluster barrier per exchange; a digit round's counts
// alternate between two buffers, so that a round needs one barrier.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "device_common.cuh"
#include "internal.h"

namespace rolekv {
namespace {

constexpr int kR = ROLEKV_MAX_ROLES;
constexpr uint32_t kCodeKeep = 0x40;   // the token's bucket keeps everything
constexpr uint32_t kCodeDrop = 0x80;   // no bucket keeps the token
// codes 0 .. kR-1: the token's bucket keeps only keys above a threshold
constexpr int kMaxRanks = 8;           // CTAs per unit (the portable cluster size)
constexpr int kDenseWords = 400;       // kept of 32 words above which a lane takes a slot, not an output
constexpr int kRankCost = 3000;        // most compares (sum of squared runs) taken by rank
constexpr int kTieCap = 256;           // ranked ties held in shared memory

// Launch plan of one call: ranks and threads per unit, and the layout of a
// rank's shared memory.
struct SelectPlan {
  int32_t ranks;       // CTAs per unit (the cluster size)
  int32_t nb;          // first-digit bits
  int32_t groups;      // groups (of four slots) a rank's memory holds
  int32_t n_hist;      // buckets with a histogram
  int32_t list_cap;    // candidate-list entries (8 bytes each in streaming mode, else 4)
  int32_t hist_off;    // byte offset, after keys and keep bits, of
  int32_t hist_ints;   // the two digit-count buffers (and the first-digit sums)
  int32_t region_words;   // pass-1 histograms, then the candidate list
};

// Monotone map of a float to uint32 (larger float -> larger key); -0 is folded
// onto +0 so equal floats give equal keys.
__device__ __forceinline__ uint32_t ordered_key(float f) {
  if (f == 0.0f) f = 0.0f;
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Distributed shared memory: the address of a local shared object in rank
// `rank` of the cluster, and accesses through such an address.
__device__ __forceinline__ uint32_t map_rank(const void* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ int32_t ld_rank(uint32_t addr) {
  int32_t v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ int4 ld_rank4(uint32_t addr) {
  int4 v;
  asm volatile("ld.shared::cluster.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ void st_rank(uint32_t addr, int32_t v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void add_rank(uint32_t addr, int32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Barrier over the unit's CTAs (the whole cluster), or the CTA alone.
template <bool CL>
__device__ __forceinline__ void unit_sync() {
  if constexpr (CL) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                     : "memory");
  } else {
    __syncthreads();
  }
}

// x << n, 0 for n > 63.
__device__ __forceinline__ uint64_t shl64(uint64_t x, uint32_t n) {
  uint64_t r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
}

__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct SelShared {
  // this rank's share, read by the other ranks after a barrier
  int32_t l_count[kR];     // tokens per role (GLOBAL: the eligible ones, in [0])
  int32_t l_floor[kR];     // recency-floor tokens per role
  int32_t l_nan;           // a sum of the slice's scores was NaN
  uint32_t l_and, l_or;    // of the slice's keys
  int32_t l_ties[kR];      // keys equal to a partial bucket's threshold
  int32_t l_fill_ties;     // the same for the SLACK fill
  int32_t l_total;         // kept slots
  // first digits found by other ranks (written by them, taken over after a barrier)
  uint32_t f_prefix[kR];
  int32_t f_need[kR], f_cand[kR];
  int32_t f_fail;
  // the unit's state, the same in every rank
  int64_t keep_off;
  int32_t count[kR];       // tokens per role
  int32_t quota[kR];       // q_b per bucket
  uint32_t prefix[kR];     // threshold key bits found so far
  int32_t need[kR];        // tokens equal to the prefix still to keep
  uint32_t thr[kR];        // keep iff key >= thr (ties ranked apart when partial)
  int32_t mode[kR];        // 0 none kept, 1 all kept, 2 threshold
  int32_t cand[kR];        // candidates after the first digit
  int32_t code_of_role[256];
  int32_t first_of_role[256];  // pass 2: keep iff first digit > it, candidate iff ==
  int32_t floor_role[kR];  // recency-floor tokens per role
  uint32_t top_and, top_or;
  int32_t nan_hint;        // a sum of the unit's scores was NaN
  int32_t any_threshold;
  int32_t general;         // take the full-pass descent
  uint32_t partial_ties;   // buckets with more threshold ties than slots left
  int32_t slack;           // SLACK policy: slots left to fill by score
  uint32_t elig_mask;      // roles taking part in the split (bit r)
  int32_t sfast;           // SLACK: the fill's first digit is known (below)
  uint32_t sprefix;        // SLACK: shared top bit and first digit of the fill threshold
  int32_t sneed;           // SLACK: tokens at that digit still to fill
  // this rank's own
  int32_t warp_tot[32];
  int32_t kept_role[kR];   // (rank 0: the ranks add to it)
  uint32_t ties[kTieCap];  // (bucket << 16) | slot of keys equal to a threshold
  int32_t list_n, tie_n;
  int32_t run0[kR], run_n[kR];   // candidate runs of the buckets
  int32_t nan_seen;        // a pooled window held a NaN
};

// Slots 4g .. 4g+3 of a score row; slots outside [off, off + n) read -inf.
// sp + (4g - off) is 16-byte aligned by the choice of off.  ORDERED: the load
// is issued where it stands, together with its neighbours' (8 rows of 512
// tokens 8.2 us, 8.4 as the compiler places plain loads; streaming mode, which
// drops the loads its pool does not need, is 2% faster with those).
template <bool ORDERED>
__device__ __forceinline__ float4 load_slots(const float* sp, int off, int n, int g) {
  const int s0 = 4 * g - off;
  if (s0 >= 0 && s0 + 4 <= n) {
    if (!ORDERED) return *reinterpret_cast<const float4*>(sp + s0);
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(sp + s0));
    return v;
  }
  float4 r;
  r.x = (s0 >= 0 && s0 < n) ? sp[s0] : -INFINITY;
  r.y = (s0 + 1 >= 0 && s0 + 1 < n) ? sp[s0 + 1] : -INFINITY;
  r.z = (s0 + 2 >= 0 && s0 + 2 < n) ? sp[s0 + 2] : -INFINITY;
  r.w = (s0 + 3 >= 0 && s0 + 3 < n) ? sp[s0 + 3] : -INFINITY;
  return r;
}

// Role bytes of slots 4g .. 4g+3 (0xFF outside the sequence).
__device__ __forceinline__ uint32_t load_roles(const uint8_t* rp, int off, int n, int g, bool vec) {
  const int s0 = 4 * g - off;
  if (vec && s0 >= 0 && s0 + 4 <= n) return *reinterpret_cast<const uint32_t*>(rp + s0);
  uint32_t w = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int t = s0 + j;
    const uint32_t r = (t >= 0 && t < n) ? static_cast<uint32_t>(rp[t]) : 0xFFu;
    w |= r << (8 * j);
  }
  return w;
}

struct UnitView {
  const float* sp;
  const uint8_t* rp;
  int off, n;
  int g0, ng;      // this rank's groups: g0 .. g0 + ng - 1
  int nf;          // tokens before the recency floor (the floor is [nf, n))
  bool rvec;
};

// Bits j of the slots 4g+j (first token s0 = 4g - off) inside the recency
// floor [nf, n).
__device__ __forceinline__ uint32_t floor_bits(int s0, int nf, int n) {
  if (s0 + 4 <= nf || s0 >= n) return 0u;
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (s0 + j >= nf && s0 + j < n) m |= 1u << j;
  return m;
}

// Pass 1 over the rank's groups for a pool half-width HW known at compile
// time; floor tokens are counted apart.
template <int HW, int NT, bool GL, bool STREAM>
__device__ __forceinline__ void pass1(const UnitView& v, int n_roles, uint32_t ban, int nb,
                                      uint4* keys4, uint32_t* hist16, int32_t* floor_role,
                                      bool& nan_hint, uint32_t& top_and, uint32_t& top_or) {
  constexpr int NB = (HW + 3) / 4;   // neighbour groups on each side
  const int sh0 = 31 - nb;
  const uint32_t bmask = (1u << nb) - 1u;
  const int words_per_role = 1 << (nb - 1);
  for (int lg = threadIdx.x; lg < v.ng; lg += NT) {
    const int g = v.g0 + lg;
    // the role bytes are loaded with the scores, not after the pooling
    const uint32_t rw = load_roles(v.rp, v.off, v.n, g, v.rvec);
    float x[4 * (2 * NB + 1)];
#pragma unroll
    for (int o = -NB; o <= NB; ++o) {
      const float4 f = load_slots<!STREAM>(v.sp, v.off, v.n, g + o);
      x[4 * (o + NB) + 0] = f.x;
      x[4 * (o + NB) + 1] = f.y;
      x[4 * (o + NB) + 2] = f.z;
      x[4 * (o + NB) + 3] = f.w;
    }
    const float* c = x + 4 * NB;
    const float sum = (c[0] + c[1]) + (c[2] + c[3]);
    nan_hint |= (sum != sum);
    uint32_t k[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float m = c[j - HW];
#pragma unroll
      for (int o = -HW + 1; o <= HW; o += 2) {
        if (o < HW)
          m = max3f(m, c[j + o], c[j + o + 1]);
        else
          m = fmaxf(m, c[j + o]);
      }
      k[j] = ordered_key(m);
    }
    if (!STREAM) keys4[lg] = make_uint4(k[0], k[1], k[2], k[3]);
    const uint32_t fb = floor_bits(4 * g - v.off, v.nf, v.n);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t r = (rw >> (8 * j)) & 0xFFu;
      if ((fb >> j) & 1u) {                      // recency floor: kept, counted apart
        if (r < static_cast<uint32_t>(n_roles)) atomicAdd(&floor_role[r], 1);
      } else if (r < static_cast<uint32_t>(n_roles)) {
        top_and &= k[j];
        top_or |= k[j];
        const uint32_t bin = (k[j] >> sh0) & bmask;
        if (!GL || !((ban >> r) & 1u)) {
          if (STREAM)
            atomicAdd(&hist16[((GL ? 0u : r) << nb) + bin], 1u);   // 32-bit bins
          else
            atomicAdd(&hist16[(GL ? 0u : r) * words_per_role + (bin >> 1)], 1u << (16 * (bin & 1u)));
        }
      }
    }
  }
}

// Quotas of one sequence by warp 0, lane r for role r: water-filling of the
// weights over the role counts, then the integer remainders to the largest
// fractional parts (ties to the lower role), or under CEIL the ceiling of each
// share; the arithmetic stated in rolekv.h.
__device__ __forceinline__ int64_t sum8(int64_t v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  return v;
}

// Streaming mode: the four keys of group g recomputed from the score row, the
// same max-pool as pass 1 (stride 1, -inf outside the row, half-width hw);
// nan_aware: a window holding a NaN gives key 0 (below every other key).
__device__ __forceinline__ uint4 stream_group_keys(const UnitView& v, int g, int hw, bool nan_aware) {
  float x[20];
#pragma unroll
  for (int o = -2; o <= 2; ++o) {
    const float4 f = load_slots<false>(v.sp, v.off, v.n, g + o);
    x[4 * (o + 2) + 0] = f.x;
    x[4 * (o + 2) + 1] = f.y;
    x[4 * (o + 2) + 2] = f.z;
    x[4 * (o + 2) + 3] = f.w;
  }
  uint32_t k[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float m = x[8 + j];
    bool nanw = m != m;
#pragma unroll
    for (int d = 1; d <= 7; ++d) {
      if (d <= hw) {
        const float lo = x[8 + j - d], hi = x[8 + j + d];
        nanw |= (lo != lo) | (hi != hi);
        m = max3f(m, lo, hi);
      }
    }
    k[j] = (nan_aware && nanw) ? 0u : ordered_key(m);
  }
  return make_uint4(k[0], k[1], k[2], k[3]);
}

__device__ void quotas_warp(const SelectArgs& a, int lane, int64_t K_full, SelShared& S) {
  // every group of 8 lanes holds the 8 roles, so sums over a group are the
  // totals and all lanes take the same branches
  const int r = lane & (kR - 1);
  const bool valid = r < a.n_roles;
  const bool banned = valid && ((a.ban_mask >> r) & 1u);
  const int64_t cnt = valid ? S.count[r] : 0;
  // FAIR: every non-banned role weighted by its own token count
  const int64_t alpha = (a.policy == ROLEKV_POLICY_FAIR) ? ((valid && !banned) ? cnt : 0)
                                                         : a.alpha_fx[r];
  int64_t q = 0, bsize = 0;
  if (a.policy == ROLEKV_POLICY_GLOBAL) {
    const int64_t elig = S.count[0];   // every eligible token, counted in row 0
    if (r == 0) {
      q = K_full < elig ? K_full : elig;
      bsize = elig;
    }
  } else {
    bool live = valid && alpha > 0 && cnt > 0;
    const unsigned elig_bits = __ballot_sync(0xffffffffu, live) & 0xFFu;
    const int64_t elig = sum8(live ? cnt : 0);
    const int64_t k_all = K_full < elig ? K_full : elig;
    int64_t left = k_all;
    // SLACK: one round of the split, no water-filling (the slack of saturated
    // buckets is filled by score afterwards)
    for (int it = 0; it <= kR && a.policy != ROLEKV_POLICY_SLACK; ++it) {
      const int64_t A = sum8(live ? alpha : 0);
      if (A == 0) break;
      const bool sat = live && alpha * left >= cnt * A;
      if (!__any_sync(0xffffffffu, sat)) break;
      if (sat) {
        q = cnt;
        live = false;
      }
      left -= sum8(sat ? cnt : 0);
    }
    const int64_t A = sum8(live ? alpha : 0);
    if (a.policy == ROLEKV_POLICY_CEIL) {
      // Algorithm 1 read literally: each unsaturated bucket takes the ceiling
      // of its share (the total may exceed the budget; the rows are wider)
      if (live && A != 0) q = (alpha * left + A - 1) / A;
    } else {
      int64_t rem = -1;
      if (live && A != 0) {
        q = alpha * left / A;
        rem = alpha * left % A;
      }
      const int64_t extra = left - sum8(live ? q : 0);
      int rank = 0;
#pragma unroll
      for (int x = 0; x < kR; ++x) {
        const int64_t rx = __shfl_sync(0xffffffffu, rem, x);
        const int lx = __shfl_sync(0xffffffffu, static_cast<int>(live), x);
        if (lx && (rx > rem || (rx == rem && x < r))) ++rank;
      }
      if (live && A != 0 && rank < extra) q += 1;
    }
    if (a.policy == ROLEKV_POLICY_SLACK) {
      q = q < cnt ? q : cnt;
      const int64_t slack = k_all - sum8(q);
      if (lane == 0) {
        S.slack = static_cast<int32_t>(slack);
        S.elig_mask = elig_bits;
      }
    }
    bsize = cnt;
  }
  int mode = 0;
  if (lane < kR) {
    mode = (q <= 0) ? 0 : (q >= bsize ? 1 : 2);
    S.quota[r] = static_cast<int32_t>(q);
    S.mode[r] = mode;
    S.prefix[r] = 0;
    S.need[r] = static_cast<int32_t>(q);
    S.thr[r] = 0xFFFFFFFFu;   // above every key; set by the last radix round
    S.cand[r] = 0;
  }
  const bool any = __any_sync(0xffffffffu, mode == 2);
  if (lane == 0) {
    S.any_threshold = any;
    S.partial_ties = 0;
    S.list_n = 0;
    S.tie_n = 0;
  }
}

// The bucket's key among its remaining candidates with need[b] keys at or
// above it: one warp sums the ranks' counts of the digit at `shift` (hist),
// finds the digit where the count from the top reaches need[b], appends it to
// prefix[b] and subtracts the keys above.  At shift 0 the prefix is the
// q_b-th largest key; thr[b] and the partial-tie flag are then set.  Every
// rank does it alike.
template <bool CL>
__device__ void descend(SelShared& S, const int32_t* hist, int ranks, int b, int lane, int shift) {
  int c[8];
  const int32_t* hb = hist + b * 256 + lane * 8;
  if constexpr (CL) {
#pragma unroll
    for (int i = 0; i < 8; ++i) c[i] = 0;
    // (four ranks' loads in flight)
    for (int k0 = 0; k0 < ranks; k0 += 4) {
      int4 x[4], y[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k0 + k < ranks) {
          const uint32_t addr = map_rank(hb, k0 + k);
          x[k] = ld_rank4(addr);
          y[k] = ld_rank4(addr + 16);
        } else {
          x[k] = y[k] = make_int4(0, 0, 0, 0);
        }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        c[0] += x[k].x; c[1] += x[k].y; c[2] += x[k].z; c[3] += x[k].w;
        c[4] += y[k].x; c[5] += y[k].y; c[6] += y[k].z; c[7] += y[k].w;
      }
    }
  } else {
    const int4 x = *reinterpret_cast<const int4*>(hb), y = *reinterpret_cast<const int4*>(hb + 4);
    c[0] = x.x; c[1] = x.y; c[2] = x.z; c[3] = x.w;
    c[4] = y.x; c[5] = y.y; c[6] = y.z; c[7] = y.w;
  }
  int mine = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) mine += c[i];
  int incl = mine;   // tokens whose digit is in this lane's range or above
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_down_sync(0xffffffffu, incl, o);
    if (lane + o < 32) incl += v;
  }
  const int above = incl - mine;
  const int need = S.need[b];
  int found = -1, gt_before = 0, at_digit = 0;
  if (above < need && above + mine >= need) {
    int acc = above;
#pragma unroll
    for (int i = 7; i >= 0; --i) {
      if (found < 0 && acc + c[i] >= need) {
        found = lane * 8 + i;
        gt_before = acc;
        at_digit = c[i];
      }
      acc += c[i];
    }
  }
  const unsigned who = __ballot_sync(0xffffffffu, found >= 0);
  const int src = who ? __ffs(who) - 1 : 0;
  const int fd = __shfl_sync(0xffffffffu, found, src);
  const int gb = __shfl_sync(0xffffffffu, gt_before, src);
  const int ad = __shfl_sync(0xffffffffu, at_digit, src);
  if (lane == 0 && who != 0) {
    const uint32_t prefix = S.prefix[b] | (static_cast<uint32_t>(fd) << shift);
    const int need2 = need - gb;
    S.prefix[b] = prefix;
    S.need[b] = need2;
    S.cand[b] = ad;
    if (shift == 0) {
      // ad keys of the bucket equal the threshold; need2 of them are kept
      S.thr[b] = (need2 >= ad) ? prefix : prefix + 1u;
      if (need2 < ad) atomicOr(&S.partial_ties, 1u << b);
    }
  }
}

// First digit (bits 30..31-nb, the shared top bit above them) of bucket b from
// the per-role 16-bit histograms of pass 1; the bucket's histogram is the sum
// over its roles.  Lane L owns a contiguous range of bins: the lanes' totals
// (read in a rotated order, so that the lanes hit different banks) locate the
// lane holding the threshold, then the warp splits that lane's words.
template <int NB>
__device__ void descend_first(const SelectArgs& a, SelShared& S, const uint32_t* hist16, int b,
                              int lane) {
  constexpr int nb = NB;
  constexpr int wpl = 1 << (nb - 6);   // histogram words (two bins each) per lane
  constexpr int wpr = 1 << (nb - 1);   // words per role
  // counts of bins 2w (low half) and 2w+1 (high half); a bin holds at most
  // n < 65536 tokens, so the halves never carry
  const uint32_t* h0 = hist16 + b * wpr;
  int mine = 0;
#pragma unroll
  for (int i = 0; i < wpl; ++i) {
    const uint32_t x = h0[lane * wpl + ((i + lane) & (wpl - 1))];
    mine += static_cast<int>((x & 0xFFFFu) + (x >> 16));
  }
  int incl = mine;   // tokens in this lane's bins or above
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_down_sync(0xffffffffu, incl, o);
    if (lane + o < 32) incl += v;
  }
  const int above = incl - mine;
  const int need = S.need[b];
  const unsigned who = __ballot_sync(0xffffffffu, above < need && above + mine >= need);
  if (who == 0) {
    if (lane == 0) S.general = 1;   // counts disagree with the quota: let the full path decide
    return;
  }
  const int F = __ffs(who) - 1;
  const int aboveF = __shfl_sync(0xffffffffu, above, F);
  const int needF = need - aboveF;
  const uint32_t x = lane < wpl ? h0[F * wpl + lane] : 0u;
  const int lo = static_cast<int>(x & 0xFFFFu), hi = static_cast<int>(x >> 16);
  const int pair = lo + hi;
  int incl2 = pair;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_down_sync(0xffffffffu, incl2, o);
    if (lane + o < 32) incl2 += v;
  }
  const int above2 = incl2 - pair;
  const unsigned who2 = __ballot_sync(0xffffffffu, above2 < needF && above2 + pair >= needF);
  if (who2 == 0) {
    if (lane == 0) S.general = 1;
    return;
  }
  if (lane == __ffs(who2) - 1) {
    const int w = F * wpl + lane;
    int fd, gb, ad;
    if (above2 + hi >= needF) {
      fd = 2 * w + 1;
      gb = aboveF + above2;
      ad = hi;
    } else {
      fd = 2 * w;
      gb = aboveF + above2 + hi;
      ad = lo;
    }
    const int sh0 = 31 - nb;
    S.prefix[b] = (S.top_and & 0x80000000u) | (static_cast<uint32_t>(fd) << sh0);
    S.need[b] = need - gb;
    S.cand[b] = ad;
  }
}

// SLACK policy: the first digit of the fill threshold, from the same pass-1
// histograms, once every bucket's first digit is known.  The tokens the fill
// ranks are the eligible ones no bucket keeps; per first-digit bin they are
// a role's whole bin (its bucket keeps nothing, or the bin lies below the
// bucket's digit), none (the bucket keeps the bin), or the bin less the
// need[b] tokens the bucket keeps at its own digit.  Every thread counts a
// few bins of its rank into `cnt` (shared memory, 2^NB ints); rank 0 adds the
// ranks' counts, and its warp 0 locates the bin holding the slack-th token
// from the top: each lane sums a contiguous range, the lanes' totals from the
// top locate the range, and the warp splits that range.  On success sprefix /
// sneed are set and sfast = 1 in every rank; otherwise the fill takes its
// full-pass rounds.  cnt is left with counts in it.
template <int NB, int NT, bool CL>
__device__ void slack_first(const SelectArgs& a, SelShared& S, const uint32_t* hist16, int* cnt,
                            int list_cap, int slice_slots, int rank, int ranks) {
  constexpr int nbins = 1 << NB;
  constexpr int bpl = nbins / 32;        // bins per lane
  constexpr int wpr = 1 << (NB - 1);     // histogram words (two bins each) per role
  constexpr int sh0 = 31 - NB;
  const int tid = threadIdx.x, lane = tid & 31;
  for (int x = tid; x < nbins; x += NT) {
    int c = 0;
    for (int r = 0; r < a.n_roles; ++r) {
      if (!((S.elig_mask >> r) & 1u)) continue;
      const uint32_t code = static_cast<uint32_t>(S.code_of_role[r]);
      if (code == kCodeKeep) continue;
      const uint32_t w = hist16[r * wpr + (x >> 1)];
      const int h = static_cast<int>((x & 1) ? (w >> 16) : (w & 0xFFFFu));
      if (code >= static_cast<uint32_t>(kR)) {
        c += h;                                  // its bucket keeps nothing
      } else {
        const int D = static_cast<int>((S.prefix[code] >> sh0) & (nbins - 1));
        // (the need[b] tokens are the unit's: taken off once, in rank 0)
        c += x < D ? h : (x == D ? h - (rank == 0 ? S.need[code] : 0) : 0);
      }
    }
    cnt[x] = c;
  }
  unit_sync<CL>();
  if (rank == 0) {
    if constexpr (CL) {
      for (int x = tid; x < nbins; x += NT) {
        int c[kMaxRanks];
#pragma unroll
        for (int k = 0; k < kMaxRanks; ++k) c[k] = k < ranks ? ld_rank(map_rank(cnt + x, k)) : 0;
#pragma unroll
        for (int k = 1; k < kMaxRanks; ++k) c[0] += c[k];
        cnt[x] = c[0];
      }
      __syncthreads();
    }
    if (warp_uniform(tid >> 5) == 0) {
      const int need = S.slack;
      int mine = 0;
#pragma unroll 8
      for (int i = 0; i < bpl; ++i) mine += cnt[lane * bpl + ((i + lane) & (bpl - 1))];
      int incl = mine;                             // tokens in this lane's bins or above
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_down_sync(0xffffffffu, incl, o);
        if (lane + o < 32) incl += v;
      }
      const int above = incl - mine;
      const unsigned who = __ballot_sync(0xffffffffu, above < need && above + mine >= need);
      if (who != 0) {
        const int F = __ffs(who) - 1;
        const int aboveF = __shfl_sync(0xffffffffu, above, F);
        const int needF = need - aboveF;
        // the winning range split over the warp: bpl / 32 bins a lane
        constexpr int per = bpl / 32 > 0 ? bpl / 32 : 1;
        int c2[per];
        int part = 0;
#pragma unroll
        for (int i = 0; i < per; ++i) {
          c2[i] = (lane * per + i < bpl) ? cnt[F * bpl + lane * per + i] : 0;
          part += c2[i];
        }
        int incl2 = part;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_down_sync(0xffffffffu, incl2, o);
          if (lane + o < 32) incl2 += v;
        }
        const int above2 = incl2 - part;
        const unsigned who2 = __ballot_sync(0xffffffffu, above2 < needF && above2 + part >= needF);
        if (who2 != 0 && lane == __ffs(who2) - 1) {
          int acc = above2, fd = -1, nd = 0, at = 0;
#pragma unroll
          for (int i = per - 1; i >= 0; --i) {
            if (fd < 0 && acc + c2[i] >= needF) {
              fd = F * bpl + lane * per + i;
              nd = needF - acc;
              at = c2[i];
            }
            acc += c2[i];
          }
          if (fd >= 0 && (at <= list_cap || slice_slots <= list_cap)) {
            const uint32_t prefix = (S.top_and & 0x80000000u) | (static_cast<uint32_t>(fd) << sh0);
            if constexpr (CL) {
              for (int k = 0; k < ranks; ++k) {
                st_rank(map_rank(&S.sprefix, k), static_cast<int32_t>(prefix));
                st_rank(map_rank(&S.sneed, k), nd);
                st_rank(map_rank(&S.sfast, k), 1);
              }
            } else {
              S.sprefix = prefix;
              S.sneed = nd;
              S.sfast = 1;
            }
          }
        }
      }
    }
  }
  unit_sync<CL>();
}

// descend_first over the ranks' summed counts (32-bit bins, `sums`), by one
// warp; the result goes to every rank.  Lane L owns bins L * 2^NB / 32 ..; the
// lanes' totals locate the lane holding the threshold, then the warp splits
// that lane's bins (at most 64, two per lane).
template <int NB>
__device__ void descend_first_sums(SelShared& S, const int32_t* sums, int b, int lane, int ranks) {
  constexpr int bpl = 1 << (NB - 5);   // bins per lane
  int mine = 0;
#pragma unroll 8
  for (int i = 0; i < bpl; ++i) mine += sums[lane * bpl + ((i + lane) & (bpl - 1))];
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_down_sync(0xffffffffu, incl, o);
    if (lane + o < 32) incl += v;
  }
  const int above = incl - mine;
  const int need = S.need[b];
  const unsigned who = __ballot_sync(0xffffffffu, above < need && above + mine >= need);
  const int F = who ? __ffs(who) - 1 : 0;
  const int aboveF = __shfl_sync(0xffffffffu, above, F);
  const int needF = need - aboveF;
  // lane L takes bins F * bpl + 2L, 2L + 1 (descending order: the higher bin first)
  const int i0 = 2 * lane;
  const int lo = i0 < bpl ? sums[F * bpl + i0] : 0;
  const int hi = i0 + 1 < bpl ? sums[F * bpl + i0 + 1] : 0;
  const int pair = lo + hi;
  int incl2 = pair;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_down_sync(0xffffffffu, incl2, o);
    if (lane + o < 32) incl2 += v;
  }
  const int above2 = incl2 - pair;
  const unsigned who2 = __ballot_sync(0xffffffffu, above2 < needF && above2 + pair >= needF);
  const int src = who2 ? __ffs(who2) - 1 : 0;
  const bool upper = above2 + hi >= needF;
  const int fd = __shfl_sync(0xffffffffu, F * bpl + i0 + (upper ? 1 : 0), src);
  const int gb = __shfl_sync(0xffffffffu, aboveF + above2 + (upper ? 0 : hi), src);
  const int ad = __shfl_sync(0xffffffffu, upper ? hi : lo, src);
  if (lane < ranks) {
    if (who == 0 || who2 == 0) {
      st_rank(map_rank(&S.f_fail, lane), 1);   // counts disagree with the quota: the full path decides
    } else {
      const uint32_t prefix = (S.top_and & 0x80000000u) | (static_cast<uint32_t>(fd) << (31 - NB));
      st_rank(map_rank(&S.f_prefix[b], lane), static_cast<int32_t>(prefix));
      st_rank(map_rank(&S.f_need[b], lane), need - gb);
      st_rank(map_rank(&S.f_cand[b], lane), ad);
    }
  }
}

// popc(mask_of(q)) summed over the bit words q < nwords: warp w walks a
// contiguous range of words; the warps' totals are left in warp_tot for
// scan_words.  Returns the total.  Every thread of the CTA calls it.
template <int NT, class MaskF>
__device__ int count_words(int nwords, MaskF mask_of, int32_t* warp_tot) {
  constexpr int NW = NT / 32;
  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int wseg = (nwords + NW - 1) / NW;
  const int q_begin = warp * wseg;
  const int q_end = min(nwords, q_begin + wseg);
  int tot = 0;
  for (int q0 = q_begin; q0 < q_end; q0 += 32) {
    const int q = q0 + lane;
    if (q < q_end) tot += __popc(mask_of(q));
  }
  tot = warp_sum(tot);
  if (lane == 0) warp_tot[warp] = tot;
  __syncthreads();
  return warp_sum(lane < NW ? warp_tot[lane] : 0);
}

// After count_words: body(q, mask, rank of the word's first set bit) once per
// word, the ranks in slot order from `base0`.
template <int NT, class MaskF, class BodyF>
__device__ void scan_words(int nwords, int base0, MaskF mask_of, BodyF body, const int32_t* warp_tot) {
  constexpr int NW = NT / 32;
  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int wseg = (nwords + NW - 1) / NW;
  const int q_begin = warp * wseg;
  const int q_end = min(nwords, q_begin + wseg);
  int base = base0 + warp_sum(lane < warp ? warp_tot[lane] : 0);
  for (int q0 = q_begin; q0 < q_end; q0 += 32) {
    const int q = q0 + lane;
    const uint32_t m = q < q_end ? mask_of(q) : 0u;
    const int c = __popc(m);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (q < q_end) body(q, m, base + incl - c);
    base += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncthreads();
}

// Keep bits of slots 4g .. 4g+3 (bit j = slot 4g+j) packed into one 32-bit
// word per 8 lanes; the lane with (lane & 7) == 0 stores word g / 8.
__device__ __forceinline__ void store_bits(uint32_t* bits, int g, int nwords, int lane, uint32_t m4) {
  uint32_t x = m4 << (4 * (lane & 7));
  x |= __shfl_xor_sync(0xffffffffu, x, 1);
  x |= __shfl_xor_sync(0xffffffffu, x, 2);
  x |= __shfl_xor_sync(0xffffffffu, x, 4);
  if ((lane & 7) == 0 && g < 8 * nwords) bits[g >> 3] = x;
}

template <int NT, int MODE>
__global__ void __launch_bounds__(NT, 1024 / NT) select_kernel(const SelectArgs a, const SelectPlan p) {
  constexpr bool CL = MODE == kCluster, STREAM = MODE == kStream;
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) uint8_t dyn[];
  __shared__ SelShared S;
  const int tid = threadIdx.x;
  const int warp = warp_uniform(tid >> 5), lane = tid & 31;
  const int ranks = CL ? p.ranks : 1;
  const int u = CL ? blockIdx.x / ranks : blockIdx.x;
  const int rank = CL ? blockIdx.x % ranks : 0;   // (clusters are consecutive blocks)
  const int h = u % a.Hkv;
  const int s = (u / a.Hkv) % a.b;
  const int l = u / (a.Hkv * a.b);
  for (int x = tid; x < p.hist_ints; x += NT)
    reinterpret_cast<int32_t*>(dyn + p.hist_off)[x] = 0;
  {
    uint4* r4 = reinterpret_cast<uint4*>(dyn + p.hist_off + static_cast<size_t>(p.hist_ints) * 4);
    const int n4 = (p.n_hist << (STREAM ? p.nb : p.nb - 1)) / 4;
    for (int x = tid; x < n4; x += NT) r4[x] = make_uint4(0u, 0u, 0u, 0u);
  }
  wait_for_previous_kernels();
  int n;
  int64_t tok0;
  if (a.varlen) {
    const int t0 = warp_uniform(a.cu_seqlens[s]);
    tok0 = t0;
    n = warp_uniform(a.cu_seqlens[s + 1]) - t0;
  } else {
    tok0 = 0;
    n = a.n_max;
  }
  const int64_t sbase =
      a.varlen ? (static_cast<int64_t>(l) * a.Hkv + h) * a.T + tok0 : static_cast<int64_t>(u) * a.n_max;
  const int64_t rbase = a.varlen ? tok0 : static_cast<int64_t>(s) * a.n_max;
  const int64_t K_s = kept_slots(n, a.budget_fx);              // the budget
  const int64_t width = kept_rows(n, a.budget_fx, a.kept_extra); // the kept row

  UnitView v;
  v.sp = a.scores + sbase;
  v.rp = a.roles + rbase;
  v.off = static_cast<int>((reinterpret_cast<uintptr_t>(v.sp) >> 2) & 3);
  v.n = n;
  const int ngroups = (v.off + n + 3) >> 2;
  const int gs = plan_groups(ngroups, ranks);       // groups a rank owns
  v.g0 = rank * gs;
  v.ng = max(0, min(ngroups - v.g0, gs));
  v.rvec = ((reinterpret_cast<uintptr_t>(v.rp) - static_cast<uintptr_t>(v.off)) & 3u) == 0;
  const int64_t n_floor = a.keep_last < n ? (a.keep_last < K_s ? a.keep_last : K_s)
                                          : (n < K_s ? n : K_s);
  v.nf = n - static_cast<int>(n_floor);
  const int off = v.off, ng = v.ng, g0 = v.g0;
  const int slot0 = 4 * g0;                         // first slot of the rank
  const int nwords = (ng + 7) >> 3;
  const int iters = (ng + NT - 1) / NT;
  const int nb = p.nb;
  // keys, keep bits, the digit counts, then the histogram / list region
  uint4* keys4 = reinterpret_cast<uint4*>(dyn);
  const uint32_t* keys = reinterpret_cast<const uint32_t*>(keys4);
  uint32_t* bits = reinterpret_cast<uint32_t*>(dyn + (STREAM ? 0 : static_cast<size_t>(p.groups) * 16));
  int32_t* hist = reinterpret_cast<int32_t*>(dyn + p.hist_off);
  uint32_t* region = reinterpret_cast<uint32_t*>(hist + p.hist_ints);
  uint32_t* hist16 = region;                    // pass 1 histograms
  uint32_t* list = region;                      // then the candidate list
  const int list_cap = p.list_cap;
  const int hsz = p.n_hist * 256;               // one digit-count buffer
  const bool global = a.policy == ROLEKV_POLICY_GLOBAL;
  const int hw = a.pool_k / 2;
  // a group's four keys: held, or recomputed from the scores
  bool nan_keys = false;                        // streaming mode: NaN windows give key 0
  auto kv_of = [&](int lg) -> uint4 {
    if constexpr (STREAM) return stream_group_keys(v, lg, hw, nan_keys);
    else return keys4[lg];
  };
  // a list entry: (bucket, slot), in streaming mode with its key before it
  constexpr int kCodeShift = STREAM ? 24 : 16;
  constexpr uint32_t kSlotMask = (1u << kCodeShift) - 1u;
  auto entry = [&](int e) { return STREAM ? list[2 * e + 1] : list[e]; };
  auto entry_key = [&](int e) { return STREAM ? list[2 * e] : keys[list[e] & kSlotMask]; };

  if (tid < kR) {
    S.l_count[tid] = 0;
    S.l_floor[tid] = 0;
    S.l_ties[tid] = 0;
    S.kept_role[tid] = 0;
  }
  if (tid == 0) {
    S.l_nan = 0;
    S.l_and = 0xFFFFFFFFu;
    S.l_or = 0u;
    S.l_fill_ties = 0;
    S.f_fail = 0;
    S.nan_seen = 0;
    S.general = 0;
    S.slack = 0;
    S.elig_mask = 0u;
    S.sfast = 0;
  }
  // ---- offset of this unit's kept row (warp 0)
  if (warp == 0) {
    int64_t off_kept = static_cast<int64_t>(u) * a.K_dense;
    if (a.varlen) {
      int64_t part = 0;
      for (int x = lane; x < s; x += 32)
        part += kept_rows(a.cu_seqlens[x + 1] - a.cu_seqlens[x], a.budget_fx, a.kept_extra);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      off_kept = (static_cast<int64_t>(l) * a.Hkv + h) * a.Ktot + part;
    }
    if (lane == 0) S.keep_off = off_kept;
  }
  __syncthreads();

  // Checked build: the unit's score row (and mask row), role row, kept row
  // and per-role counts lie inside the extents the call's shapes give, or the
  // whole unit is skipped (by all its ranks alike, before the first exchange).
#ifdef ROLEKV_CHECKED
  if (!(in_bounds(sbase, n, a.ext_scores, nullptr) && in_bounds(rbase, n, a.ext_roles, nullptr) &&
        in_bounds(S.keep_off, width, a.ext_keep, nullptr) &&
        (a.kept_per_role == nullptr ||
         in_bounds(static_cast<int64_t>(u) * a.n_roles, a.n_roles, static_cast<int64_t>(a.n_units) * a.n_roles,
                   nullptr)))) {
    if (tid == 0 && a.status != nullptr) atomicOr(a.status, ROLEKV_STATUS_BOUNDS);
    return;
  }
#endif

  // ---- pass 1: load, pool, key, first-digit histograms, role counts
  {
    bool nan_hint = false;
    uint32_t tand = 0xFFFFFFFFu, tor = 0u;
    // GLOBAL: one histogram (row 0) of every eligible token; otherwise one
    // row per role
#define ROLEKV_PASS1(HWV)                                                                           \
  (global ? pass1<HWV, NT, true, STREAM>(v, a.n_roles, a.ban_mask, nb, keys4, hist16, S.l_floor, nan_hint,  \
                                 tand, tor)                                                         \
          : pass1<HWV, NT, false, STREAM>(v, a.n_roles, a.ban_mask, nb, keys4, hist16, S.l_floor, nan_hint, \
                                  tand, tor))
    switch (a.pool_k >> 1) {
      case 0: ROLEKV_PASS1(0); break;
      case 1: ROLEKV_PASS1(1); break;
      case 2: ROLEKV_PASS1(2); break;
      case 3: ROLEKV_PASS1(3); break;
      case 4: ROLEKV_PASS1(4); break;
      case 5: ROLEKV_PASS1(5); break;
      case 6: ROLEKV_PASS1(6); break;
      default: ROLEKV_PASS1(7); break;
    }
#undef ROLEKV_PASS1
    tand = __reduce_and_sync(0xffffffffu, tand);
    tor = __reduce_or_sync(0xffffffffu, tor);
    const bool nh = __any_sync(0xffffffffu, nan_hint);
    if (lane == 0) {
      atomicAnd(&S.l_and, tand);
      atomicOr(&S.l_or, tor);
      if (nh) S.l_nan = 1;
    }
  }
  __syncthreads();
  // Role counts: the sums of the roles' histograms, a warp per role; GLOBAL:
  // the eligible total, in count[0].
  for (int r = warp; r < p.n_hist; r += NW) {
    const int w4 = STREAM ? 1 << (nb - 2) : 1 << (nb - 3);   // 16-byte words per role
    const uint4* h4 = reinterpret_cast<const uint4*>(hist16) + r * w4;
    uint32_t c = 0;
#pragma unroll 4
    for (int x = lane; x < w4; x += 32) {
      const uint4 w = h4[x];
      if (STREAM) {
        c += (w.x + w.y) + (w.z + w.w);
      } else {
        c += (w.x & 0xFFFFu) + (w.x >> 16) + (w.y & 0xFFFFu) + (w.y >> 16);
        c += (w.z & 0xFFFFu) + (w.z >> 16) + (w.w & 0xFFFFu) + (w.w >> 16);
      }
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) S.l_count[r] = static_cast<int32_t>(c);
  }
  unit_sync<CL>();

  // ---- the unit's counts, quotas (in every rank alike)
  if (warp == 0) {
    int c = 0, f = 0, nan = 0;
    uint32_t vand = 0xFFFFFFFFu, vor = 0u;
    const int r = lane & (kR - 1);
    if constexpr (CL) {
      // lanes 8 j .. 8 j + 7 read ranks j and j + 4
      int cc[2], ff[2], na[2];
      uint32_t va[2], vo[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int k = (lane >> 3) + 4 * i;
        const bool in = k < ranks;
        const int kk = in ? k : rank;
        cc[i] = ld_rank(map_rank(&S.l_count[r], kk));
        ff[i] = ld_rank(map_rank(&S.l_floor[r], kk));
        na[i] = ld_rank(map_rank(&S.l_nan, kk));
        va[i] = static_cast<uint32_t>(ld_rank(map_rank(&S.l_and, kk)));
        vo[i] = static_cast<uint32_t>(ld_rank(map_rank(&S.l_or, kk)));
        if (!in) {
          cc[i] = 0;
          ff[i] = 0;
        }
      }
      c = cc[0] + cc[1];
      f = ff[0] + ff[1];
      c += __shfl_xor_sync(0xffffffffu, c, 8);
      c += __shfl_xor_sync(0xffffffffu, c, 16);
      f += __shfl_xor_sync(0xffffffffu, f, 8);
      f += __shfl_xor_sync(0xffffffffu, f, 16);
      nan = __any_sync(0xffffffffu, na[0] | na[1]);
      vand = __reduce_and_sync(0xffffffffu, va[0] & va[1]);
      vor = __reduce_or_sync(0xffffffffu, vo[0] | vo[1]);
    } else {
      c = S.l_count[r];
      f = S.l_floor[r];
      nan = S.l_nan;
      vand = S.l_and;
      vor = S.l_or;
    }
    if (lane < kR) {
      S.count[lane] = c;
      S.floor_role[lane] = f;
    }
    if (lane == 0) {
      S.nan_hint = nan;
      S.top_and = vand;
      S.top_or = vor;
      if (nan || ((vand ^ vor) & 0x80000000u)) S.general = 1;
    }
    __syncwarp();
    quotas_warp(a, lane, K_s - n_floor, S);
  }
  __syncthreads();

  // A NaN score (or +inf and -inf in one group): redo the keys one token at a
  // time, a window holding a NaN giving the lowest key (streaming mode: every
  // later recomputation of the keys does so).
  nan_keys = S.nan_hint != 0;
  if (S.nan_hint) {
    uint32_t* kw = reinterpret_cast<uint32_t*>(keys4);
    bool seen = false;
    for (int t = max(0, slot0 - off) + tid; t < min(n, slot0 + 4 * ng - off); t += NT) {
      const int lo = max(0, t - (STREAM ? 0 : hw)), hi = min(n - 1, t + (STREAM ? 0 : hw));
      float m = v.sp[lo];
      bool nan_w = isnan(m);
      for (int x = lo + 1; x <= hi; ++x) {
        const float f = v.sp[x];
        nan_w |= isnan(f);
        m = fmaxf(m, f);
      }
      seen |= nan_w;
      if (!STREAM) kw[t + off - slot0] = nan_w ? 0u : ordered_key(m);
    }
    if (__any_sync(0xffffffffu, seen) && lane == 0) S.nan_seen = 1;
  }

  // ---- the role -> code table
  for (int x = tid; x < 256; x += NT) {
    uint32_t code = kCodeDrop;
    if (x < a.n_roles && !((a.ban_mask >> x) & 1u)) {
      const int b = (a.policy == ROLEKV_POLICY_GLOBAL) ? 0 : x;
      code = S.mode[b] == 2 ? static_cast<uint32_t>(b) : (S.mode[b] == 1 ? kCodeKeep : kCodeDrop);
    }
    S.code_of_role[x] = static_cast<int32_t>(code);
  }
  const bool any_thr = warp_uniform(S.any_threshold) != 0;
  const bool try_fast = warp_uniform(S.general) == 0;            // (the same in every rank)
  __syncthreads();

  // ---- first digit per bucket
  if (any_thr && try_fast) {
    if constexpr (CL) {
      // bucket b by rank b mod C, over the ranks' summed histograms
      for (int b = rank; b < p.n_hist; b += ranks) {
        if (warp_uniform(S.mode[b]) != 2) continue;
        const int wpr = 1 << (nb - 1);
        for (int x = tid; x < wpr / 4; x += NT) {
          int c[8] = {0, 0, 0, 0, 0, 0, 0, 0};
          int4 v4[kMaxRanks];                      // (all ranks' loads in flight)
#pragma unroll
          for (int k = 0; k < kMaxRanks; ++k)
            v4[k] = k < ranks ? ld_rank4(map_rank(hist16 + b * wpr + 4 * x, k)) : make_int4(0, 0, 0, 0);
#pragma unroll
          for (int k = 0; k < kMaxRanks; ++k) {
            const int4 w = v4[k];
            c[0] += w.x & 0xFFFF; c[1] += static_cast<uint32_t>(w.x) >> 16;
            c[2] += w.y & 0xFFFF; c[3] += static_cast<uint32_t>(w.y) >> 16;
            c[4] += w.z & 0xFFFF; c[5] += static_cast<uint32_t>(w.z) >> 16;
            c[6] += w.w & 0xFFFF; c[7] += static_cast<uint32_t>(w.w) >> 16;
          }
          reinterpret_cast<int4*>(hist)[2 * x] = make_int4(c[0], c[1], c[2], c[3]);
          reinterpret_cast<int4*>(hist)[2 * x + 1] = make_int4(c[4], c[5], c[6], c[7]);
        }
        __syncthreads();
        if (warp == 0) {
          if (nb == 11)
            descend_first_sums<11>(S, hist, b, lane, ranks);
          else
            descend_first_sums<10>(S, hist, b, lane, ranks);
        }
        __syncthreads();
      }
    } else {
      for (int b = warp; b < p.n_hist; b += NW) {
        if (warp_uniform(S.mode[b]) != 2) continue;
        if (STREAM)
          descend_first_sums<11>(S, reinterpret_cast<const int32_t*>(hist16) + (b << 11), b, lane, 1);
        else if (nb == 11)
          descend_first<11>(a, S, hist16, b, lane);
        else
          descend_first<10>(a, S, hist16, b, lane);
      }
    }
    if (CL || STREAM) {                            // (found by another rank, or in the sums' form)
      unit_sync<CL>();
      if (tid < p.n_hist && S.mode[tid] == 2) {
        S.prefix[tid] = S.f_prefix[tid];
        S.need[tid] = S.f_need[tid];
        S.cand[tid] = S.f_cand[tid];
      }
      if (tid == 0 && S.f_fail) S.general = 1;
    }
    __syncthreads();
  }
  // SLACK: the fill's first digit from the same histograms, before their
  // region becomes the candidate list
  const bool slack_fast = !STREAM && warp_uniform(S.slack) > 0 && warp_uniform(S.general) == 0;
  if (slack_fast) {
    if (nb == 11)
      slack_first<11, NT, CL>(a, S, hist16, hist, list_cap, 4 * gs, rank, ranks);
    else
      slack_first<10, NT, CL>(a, S, hist16, hist, list_cap, 4 * gs, rank, ranks);
  }
  if ((CL && any_thr && try_fast) || slack_fast) {
    for (int x = tid; x < p.hist_ints; x += NT) hist[x] = 0;   // (the sums above)
    __syncthreads();
  }

  // A digit round over counts the threads added to cur_hist(): the ranks meet,
  // the warps of every rank find the buckets' digits, and the other buffer
  // (read by the ranks a round ago) is cleared for the next round.
  int round_no = 0;
  auto cur_hist = [&]() { return hist + (round_no & 1) * hsz; };
  auto end_round = [&](int shift, bool fill) {
    unit_sync<CL>();
    const int32_t* H = cur_hist();
    for (int b = warp; b < (fill ? 1 : p.n_hist); b += NW)
      if (fill || warp_uniform(S.mode[b]) == 2) descend<CL>(S, H, ranks, b, lane, shift);
    ++round_no;
    int32_t* O = cur_hist();
    for (int x = tid; x < hsz; x += NT) O[x] = 0;
    __syncthreads();
  };

  // While the keys at the buckets' first digits overflow the list (scores in
  // a narrow range, such as page bounds), one full pass per 8 more bits.
  int shd = 31 - nb;   // key bits below the decided prefixes
  bool general = warp_uniform(S.general) != 0;
  if (any_thr && !general) {
    auto overflows = [&]() {
      const int t = __reduce_add_sync(0xffffffffu, lane < p.n_hist && S.mode[lane] == 2 ? S.cand[lane] : 0);
      return min(t, 4 * gs) > list_cap;
    };
    while (overflows() && shd > 8) {
      const int shift = shd - 8;
      int32_t* H = cur_hist();
      for (int i = 0; i < iters; ++i) {
        const int lg = i * NT + tid;
        if (lg >= ng) break;
        const uint4 kv = kv_of(lg);
        const uint32_t kk[4] = {kv.x, kv.y, kv.z, kv.w};
        const uint32_t rw = load_roles(v.rp, off, n, g0 + lg, v.rvec);
        const uint32_t fb = floor_bits(4 * (g0 + lg) - off, v.nf, n);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t c = static_cast<uint32_t>(S.code_of_role[(rw >> (8 * j)) & 0xFFu]);
          if (c >= static_cast<uint32_t>(kR) || ((fb >> j) & 1u)) continue;
          if ((kk[j] >> shd) != (S.prefix[c] >> shd)) continue;
          atomicAdd(&H[c * 256 + ((kk[j] >> shift) & 0xFFu)], 1);
        }
      }
      end_round(shift, false);
      shd = shift;
    }
    general = overflows();
  }

  // Ties of bucket b's threshold beyond the shared list, over the rank's
  // slots: the first `need` of the words' tie bits join the keep bits.
  auto keep_ties = [&](int need) {
    return [&bits, need](int q, uint32_t mk, int rank0) {
      uint32_t keepm = 0;
      while (mk != 0 && rank0 < need) {
        const uint32_t low = mk & (0u - mk);
        keepm |= low;
        mk ^= low;
        ++rank0;
      }
      if (keepm) bits[q] |= keepm;
    };
  };
  // need ties of the unit less those the ranks before this one hold
  auto need_here = [&](int need, const int32_t* l_ties) {
    if constexpr (CL)
      for (int k = 0; k < rank; ++k) need -= ld_rank(map_rank(l_ties, k));
    return need;
  };
  // slots of word q whose key is `key` and whose bucket is b
  auto bucket_ties = [&](int b, uint32_t key) {
    return [&, b, key](int q) {
      uint32_t mk = 0;
#pragma unroll
      for (int gg = 0; gg < 8; ++gg) {
        const int lg = 8 * q + gg;
        if (lg >= ng) break;
        const uint4 kv = kv_of(lg);
        const uint32_t kk[4] = {kv.x, kv.y, kv.z, kv.w};
        const uint32_t rw = load_roles(v.rp, off, n, g0 + lg, v.rvec);
        const uint32_t fb = floor_bits(4 * (g0 + lg) - off, v.nf, n);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (S.code_of_role[(rw >> (8 * j)) & 0xFFu] == b && kk[j] == key && !((fb >> j) & 1u))
            mk |= 1u << (4 * gg + j);
      }
      return mk;
    };
  };

  // Appends the slots of c4's bits (entries ent, keys kk) to the rank's list; the lane's
  // rank among the warp's candidates comes from four ballots.
  auto append = [&](uint32_t c4, const uint32_t* ent, const uint32_t* kk) {
    const int nc = __popc(c4);
    const unsigned b1 = __ballot_sync(0xffffffffu, nc >= 1);
    if (b1 == 0) return;
    const unsigned b2 = __ballot_sync(0xffffffffu, nc >= 2);
    const unsigned b3 = __ballot_sync(0xffffffffu, nc >= 3);
    const unsigned b4 = __ballot_sync(0xffffffffu, nc >= 4);
    const unsigned lt = (1u << lane) - 1u;
    int base = 0;
    if (lane == 0) base = atomicAdd(&S.list_n, __popc(b1) + __popc(b2) + __popc(b3) + __popc(b4));
    base = __shfl_sync(0xffffffffu, base, 0);
    int pos = base + __popc(b1 & lt) + __popc(b2 & lt) + __popc(b3 & lt) + __popc(b4 & lt);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if ((c4 >> j) & 1u) {
        if (pos < list_cap) {                      // (the counts bound the list)
          if (STREAM) {
            list[2 * pos] = kk[j];
            list[2 * pos + 1] = ent[j];
          } else {
            list[pos] = ent[j];
          }
        }
        ++pos;
      }
  };

  // Short lists (one rank): each candidate counts the candidates of its bucket
  // that come before it (larger key, or equal key and lower slot) and is kept
  // when fewer than need[b] do -- no digit rounds, no ties apart.  The list's
  // m entries are first sorted into bucket runs of cand_of(b) keys, held
  // beside the complemented slot as one 64-bit word, in the digit-count
  // buffers.  Returns false, with nothing done, when the runs are too long: 36
  // candidates in four runs take 2.4k cycles against 6.8k for three digit
  // rounds and the tie step, 274 take 10k.
  auto keep_by_rank = [&](int m, const int32_t* need, auto cand_of) {
    const int c = lane < p.n_hist ? cand_of(lane) : 0;
    int start = c;
#pragma unroll
    for (int o = 1; o < kR; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, start, o);
      if (lane >= o) start += x;
    }
    start -= c;
    const int cost = __reduce_add_sync(0xffffffffu, min(c, 1024) * min(c, 1024));
    const int total = __reduce_add_sync(0xffffffffu, c);
    if (cost > kRankCost || 2 * m > p.hist_ints || total != m) return false;
    if (warp == 0 && lane < kR) {
      S.run0[lane] = start;
      S.run_n[lane] = 0;
    }
    __syncthreads();
    uint64_t* runs = reinterpret_cast<uint64_t*>(hist);
    for (int e = tid; e < m; e += NT) {
      const uint32_t ent = list[e], b = ent >> 16, slot = ent & 0xFFFFu;
      runs[S.run0[b] + atomicAdd(&S.run_n[b], 1)] =
          (static_cast<uint64_t>(keys[slot]) << 16) | (0xFFFFu - slot);
    }
    __syncthreads();
    for (int e = tid; e < m; e += NT) {
      const uint32_t ent = list[e], b = ent >> 16, slot = ent & 0xFFFFu;
      const uint64_t mine = (static_cast<uint64_t>(keys[slot]) << 16) | (0xFFFFu - slot);
      const uint64_t* run = runs + S.run0[b];
      const int nr = S.run_n[b];
      int before = 0;
#pragma unroll 4
      for (int x = 0; x < nr; ++x) before += run[x] > mine;
      if (before < need[b]) atomicOr(&bits[slot >> 5], 1u << (slot & 31u));
    }
    __syncthreads();
    for (int x = tid; x < 2 * m; x += NT) hist[x] = 0;
    __syncthreads();
    return true;
  };

  if (!general) {
    for (int x = tid; x < 256; x += NT) {
      const uint32_t code = static_cast<uint32_t>(S.code_of_role[x]);
      S.first_of_role[x] = code == kCodeKeep                  ? -1
                           : code < static_cast<uint32_t>(kR) ? static_cast<int32_t>(S.prefix[code] >> shd)
                                                               : 0x7FFFFFFF;
    }
    __syncthreads();
    // ---- pass 2: decide every token outside its bucket's threshold digit,
    // list the rest
    // roles are read two iterations ahead of their use (they come from L2)
    auto roles_of = [&](int i) {
      const int lg = i * NT + tid;
      return (i < iters && lg < ng) ? load_roles(v.rp, off, n, g0 + lg, v.rvec) : 0xFFFFFFFFu;
    };
    uint32_t r_next = roles_of(0), r_after = roles_of(1);
    for (int i = 0; i < iters; ++i) {
      const int lg = i * NT + tid;
      const uint32_t rw = r_next;
      r_next = r_after;
      r_after = roles_of(i + 2);
      uint32_t m4 = 0, c4 = 0;
      uint32_t ent[4] = {0u, 0u, 0u, 0u};
      uint32_t kk[4] = {0u, 0u, 0u, 0u};
      if (lg < ng) {
        const uint4 kv = kv_of(lg);
        kk[0] = kv.x;
        kk[1] = kv.y;
        kk[2] = kv.z;
        kk[3] = kv.w;
        const uint32_t fb = floor_bits(4 * (g0 + lg) - off, v.nf, n);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t r = (rw >> (8 * j)) & 0xFFu;
          const int T = S.first_of_role[r];
          const int hb = static_cast<int>(kk[j] >> shd);
          m4 |= static_cast<uint32_t>(hb > T) << j;
          if (hb == T && !((fb >> j) & 1u)) {
            c4 |= 1u << j;
            ent[j] = (static_cast<uint32_t>(S.code_of_role[r]) << kCodeShift) | static_cast<uint32_t>(4 * lg + j);
          }
        }
        m4 |= fb;                                  // the recency floor is kept
      }
      store_bits(bits, lg, nwords, lane, m4);
      append(c4, ent, kk);
    }
    __syncthreads();
  }

  if (!general) {
    if (any_thr) {
      // ---- remaining bits over the candidate lists
      const int m = warp_uniform(min(S.list_n, list_cap));
      bool counted = false;
      if constexpr (MODE == kOne) counted = keep_by_rank(m, S.need, [&](int b) { return S.mode[b] == 2 ? S.cand[b] : 0; });
      for (int lo = counted ? 0 : shd; lo > 0;) {
        const int d = lo < 8 ? lo : 8;
        const int shift = lo - d;
        int32_t* H = cur_hist();
        for (int e = tid; e < m; e += NT) {
          const uint32_t c = entry(e) >> kCodeShift;
          const uint32_t key = entry_key(e);
          if ((key >> lo) == (S.prefix[c] >> lo))
            atomicAdd(&H[c * 256 + ((key >> shift) & ((1u << d) - 1u))], 1);
        }
        end_round(shift, false);
        lo = shift;
      }
      // kept candidates join the bits; ties of partial buckets are gathered
      const uint32_t partial = warp_uniform(S.partial_ties);
      for (int e = tid; e < (counted ? 0 : m); e += NT) {
        const uint32_t ent = entry(e);
        const uint32_t c = ent >> kCodeShift;
        const uint32_t slot = ent & kSlotMask;
        const uint32_t key = entry_key(e);
        if (key >= S.thr[c]) {
          atomicOr(&bits[slot >> 5], 1u << (slot & 31u));
        } else if (((partial >> c) & 1u) && key == S.prefix[c]) {
          atomicAdd(&S.l_ties[c], 1);
          const int t = atomicAdd(&S.tie_n, 1);
          if (t < kTieCap) S.ties[t] = ent;
        }
      }
      if (partial != 0) {                          // (the same in every rank)
        unit_sync<CL>();
        const int nt = warp_uniform(S.tie_n);
        if (nt <= kTieCap) {
          // index-order rank among the bucket's ties
          for (int t = tid; t < nt; t += NT) {
            const uint32_t ent = S.ties[t];
            const uint32_t c = ent >> kCodeShift, slot = ent & kSlotMask;
            int before = 0;
            for (int x = 0; x < nt; ++x) {
              const uint32_t o = S.ties[x];
              before += ((o >> kCodeShift) == c && (o & kSlotMask) < slot);
            }
            if (before < need_here(S.need[c], &S.l_ties[c])) atomicOr(&bits[slot >> 5], 1u << (slot & 31u));
          }
        } else {
          for (uint32_t pend = partial; pend != 0; pend &= pend - 1) {
            const int b = __ffs(pend) - 1;
            auto mask_of = bucket_ties(b, S.prefix[b]);
            count_words<NT>(nwords, mask_of, S.warp_tot);
            scan_words<NT>(nwords, 0, mask_of, keep_ties(need_here(S.need[b], &S.l_ties[b])), S.warp_tot);
          }
        }
      }
      __syncthreads();
    }
  } else {
    // ---- general path: four 8-bit rounds over every slot, from the top
    // (the first-digit step may have run before the list overflowed)
    if (tid < kR) {
      S.prefix[tid] = 0;
      S.need[tid] = S.quota[tid];
    }
    if (tid == 0) S.partial_ties = 0;
    __syncthreads();
    for (int round = 0; round < (any_thr ? 4 : 0); ++round) {
      const int shift = 24 - 8 * round;
      int32_t* H = cur_hist();
      for (int i = 0; i < iters; ++i) {
        const int lg = i * NT + tid;
        if (lg >= ng) break;
        const uint4 kv = kv_of(lg);
        const uint32_t kk[4] = {kv.x, kv.y, kv.z, kv.w};
        const uint32_t rw = load_roles(v.rp, off, n, g0 + lg, v.rvec);
        const uint32_t fb = floor_bits(4 * (g0 + lg) - off, v.nf, n);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t c = static_cast<uint32_t>(S.code_of_role[(rw >> (8 * j)) & 0xFFu]);
          if (c >= static_cast<uint32_t>(kR) || ((fb >> j) & 1u)) continue;
          if (round > 0 && (kk[j] >> (shift + 8)) != (S.prefix[c] >> (shift + 8))) continue;
          atomicAdd(&H[c * 256 + ((kk[j] >> shift) & 0xFFu)], 1);
        }
      }
      end_round(shift, false);
    }
    for (int i = 0; i < iters; ++i) {
      const int lg = i * NT + tid;
      uint32_t m4 = 0;
      if (lg < ng) {
        const uint4 kv = kv_of(lg);
        const uint32_t kk[4] = {kv.x, kv.y, kv.z, kv.w};
        const uint32_t rw = load_roles(v.rp, off, n, g0 + lg, v.rvec);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t c = static_cast<uint32_t>(S.code_of_role[(rw >> (8 * j)) & 0xFFu]);
          const bool keep = (c < static_cast<uint32_t>(kR)) ? (kk[j] >= S.thr[c]) : (c == kCodeKeep);
          m4 |= static_cast<uint32_t>(keep) << j;
        }
        m4 |= floor_bits(4 * (g0 + lg) - off, v.nf, n);    // the recency floor is kept
      }
      store_bits(bits, lg, nwords, lane, m4);
    }
    __syncthreads();
    // the first need[b] keys equal to the threshold, in index order
    const uint32_t partial = warp_uniform(S.partial_ties);
    for (uint32_t pend = partial; CL && pend != 0; pend &= pend - 1) {
      const int b = __ffs(pend) - 1;
      const int c = count_words<NT>(nwords, bucket_ties(b, S.prefix[b]), S.warp_tot);
      if (tid == 0) S.l_ties[b] = c;
      __syncthreads();
    }
    if (partial != 0) unit_sync<CL>();
    for (uint32_t pend = partial; pend != 0; pend &= pend - 1) {
      const int b = __ffs(pend) - 1;
      auto mask_of = bucket_ties(b, S.prefix[b]);
      count_words<NT>(nwords, mask_of, S.warp_tot);
      scan_words<NT>(nwords, 0, mask_of, keep_ties(need_here(S.need[b], &S.l_ties[b])), S.warp_tot);
    }
  }

  // ---- SLACK: the slots saturated buckets left go to the best-scoring
  // tokens of eligible roles not kept yet (ties to the lower index).  With
  // the fill's first digit known (sfast), one pass keeps such tokens above
  // it and lists those at it and the remaining bits are resolved over the
  // lists; otherwise four 8-bit rounds over all slots.  The digits go through
  // the state of bucket 0, whose own selection is complete.
  if (warp_uniform(S.slack) > 0) {
    const bool fast = warp_uniform(S.sfast) != 0;
    const uint32_t elig = S.elig_mask;
    const int sh0 = 31 - nb;
    const uint32_t bmask = (1u << nb) - 1u;
    const uint32_t DS = (S.sprefix >> sh0) & bmask;
    // an eligible slot no bucket keeps, before the recency floor
    auto candidate = [&](uint32_t rw, uint32_t fk, int j) {
      const uint32_t r = (rw >> (8 * j)) & 0xFFu;
      return r < static_cast<uint32_t>(kR) && ((elig >> r) & 1u) && !((fk >> j) & 1u);
    };
    __syncthreads();
    if (tid == 0) {
      S.list_n = 0;
      S.tie_n = 0;
      S.partial_ties = 0;
      S.prefix[0] = fast ? S.sprefix : 0u;
      S.need[0] = fast ? S.sneed : S.slack;
      S.thr[0] = 0xFFFFFFFFu;
    }
    __syncthreads();
    auto kept4 = [&](int lg) { return (bits[lg >> 3] >> (4 * (lg & 7))) & 0xFu; };
    int m = 0;
    if (fast) {
      for (int i = 0; i < iters; ++i) {
        const int lg = i * NT + tid;
        uint32_t m4 = 0, c4 = 0;
        uint32_t ent[4] = {0u, 0u, 0u, 0u};
        if (lg < ng) {
          const uint4 kv = kv_of(lg);
          const uint32_t kk[4] = {kv.x, kv.y, kv.z, kv.w};
          const uint32_t rw = load_roles(v.rp, off, n, g0 + lg, v.rvec);
          const uint32_t fk = floor_bits(4 * (g0 + lg) - off, v.nf, n) | kept4(lg);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (!candidate(rw, fk, j)) continue;
            const uint32_t d = (kk[j] >> sh0) & bmask;
            m4 |= static_cast<uint32_t>(d > DS) << j;
            c4 |= static_cast<uint32_t>(d == DS) << j;
            ent[j] = static_cast<uint32_t>(4 * lg + j);
          }
          if (m4) atomicOr(&bits[lg >> 3], m4 << (4 * (lg & 7)));
        }
        append(c4, ent, ent);                      // (held keys: not stored in the list)
      }
      __syncthreads();
      m = warp_uniform(min(S.list_n, list_cap));
      if constexpr (MODE == kOne)
        if (keep_by_rank(m, S.need, [&](int b) { return b == 0 ? m : 0; })) m = 0;
      for (int lo = m > 0 || MODE != kOne ? sh0 : 0; lo > 0;) {
        const int d = lo < 8 ? lo : 8;
        const int shift = lo - d;
        int32_t* H = cur_hist();
        for (int e = tid; e < m; e += NT) {
          const uint32_t key = keys[list[e]];
          if ((key >> lo) == (S.prefix[0] >> lo)) atomicAdd(&H[(key >> shift) & ((1u << d) - 1u)], 1);
        }
        end_round(shift, true);
        lo = shift;
      }
      const uint32_t T = S.thr[0], P = S.prefix[0];
      const bool partial = S.partial_ties & 1u;
      for (int e = tid; e < m; e += NT) {
        const uint32_t slot = list[e];
        const uint32_t key = keys[slot];
        if (key >= T) {
          atomicOr(&bits[slot >> 5], 1u << (slot & 31u));
        } else if (partial && key == P) {
          atomicAdd(&S.l_fill_ties, 1);
          const int t = atomicAdd(&S.tie_n, 1);
          if (t < kTieCap) S.ties[t] = slot;
        }
      }
      __syncthreads();
    } else {
      for (int round = 0; round < 4; ++round) {
        const int shift = 24 - 8 * round;
        int32_t* H = cur_hist();
        for (int i = 0; i < iters; ++i) {
          const int lg = i * NT + tid;
          if (lg >= ng) break;
          const uint4 kv = kv_of(lg);
          const uint32_t kk[4] = {kv.x, kv.y, kv.z, kv.w};
          const uint32_t rw = load_roles(v.rp, off, n, g0 + lg, v.rvec);
          const uint32_t fk = floor_bits(4 * (g0 + lg) - off, v.nf, n) | kept4(lg);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (!candidate(rw, fk, j)) continue;
            if (round > 0 && (kk[j] >> (shift + 8)) != (S.prefix[0] >> (shift + 8))) continue;
            atomicAdd(&H[(kk[j] >> shift) & 0xFFu], 1);
          }
        }
        end_round(shift, true);
      }
      // candidates above the threshold join
      const uint32_t T = S.thr[0];
      for (int i = 0; i < iters; ++i) {
        const int lg = i * NT + tid;
        if (lg >= ng) break;
        const uint4 kv = kv_of(lg);
        const uint32_t kk[4] = {kv.x, kv.y, kv.z, kv.w};
        const uint32_t rw = load_roles(v.rp, off, n, g0 + lg, v.rvec);
        const uint32_t fk = floor_bits(4 * (g0 + lg) - off, v.nf, n) | kept4(lg);
        uint32_t m4 = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (kk[j] >= T && candidate(rw, fk, j)) m4 |= 1u << j;
        if (m4) atomicOr(&bits[lg >> 3], m4 << (4 * (lg & 7)));
      }
      __syncthreads();
    }
    if (warp_uniform(S.partial_ties) & 1u) {       // (the same in every rank)
      const uint32_t P = S.prefix[0];
      auto mask_of = [&](int q) {
        uint32_t mk = 0;
#pragma unroll
        for (int gg = 0; gg < 8; ++gg) {
          const int lg = 8 * q + gg;
          if (lg >= ng) break;
          const uint4 kv = kv_of(lg);
          const uint32_t kk[4] = {kv.x, kv.y, kv.z, kv.w};
          const uint32_t rw = load_roles(v.rp, off, n, g0 + lg, v.rvec);
          const uint32_t fk = floor_bits(4 * (g0 + lg) - off, v.nf, n) | kept4(lg);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (kk[j] == P && candidate(rw, fk, j)) mk |= 1u << (4 * gg + j);
        }
        return mk;
      };
      if (CL && !fast) {
        const int c = count_words<NT>(nwords, mask_of, S.warp_tot);
        if (tid == 0) S.l_fill_ties = c;
      }
      unit_sync<CL>();
      const int need = need_here(S.need[0], &S.l_fill_ties);
      const int nt = warp_uniform(S.tie_n);
      if (fast && nt <= kTieCap) {
        // index-order rank among the fill's ties
        for (int t = tid; t < nt; t += NT) {
          const uint32_t slot = S.ties[t];
          int before = 0;
          for (int x = 0; x < nt; ++x) before += S.ties[x] < slot;
          if (before < need) atomicOr(&bits[slot >> 5], 1u << (slot & 31u));
        }
      } else {
        // more ties than the shared list holds: rank them over all slots
        count_words<NT>(nwords, mask_of, S.warp_tot);
        scan_words<NT>(nwords, 0, mask_of, keep_ties(need), S.warp_tot);
      }
      __syncthreads();
    }
  }

  // ---- kept positions in ascending order
  auto kept_bits = [&](int q) { return bits[q]; };
  int total = count_words<NT>(nwords, kept_bits, S.warp_tot);
  int base0 = 0;
  if constexpr (CL) {
    if (tid == 0) S.l_total = total;
    unit_sync<CL>();
    // lane k: rank k's total
    const int t = lane < ranks ? ld_rank(map_rank(&S.l_total, lane)) : 0;
    base0 = warp_sum(lane < rank ? t : 0);
    total = warp_sum(t);
  }
  int32_t* dst = a.keep_idx + S.keep_off;
  const bool count_roles = a.kept_per_role != nullptr &&
                           (a.policy == ROLEKV_POLICY_GLOBAL || a.policy == ROLEKV_POLICY_SLACK);
  // Warp w writes its words' positions, 32 words at a time, a lane per output:
  // the lane finds its word by a search over the words' prefix counts and its
  // bit by halves (a lane per word waits for the fullest word, 6.5k cycles at
  // 1024 words a CTA and a tenth kept).  Its cost grows with what is kept;
  // where that is much, a lane per slot of each word is cheaper.  512 x 8192
  // tokens, search and slots: B 0.2 41.2 and 43.8 us, 0.3 43.2 and 44.4, 0.5
  // 46.6 and 44.5; 1024 x 32768 at 0.3 223 and 231; 168 x 110545 at 0.5 229
  // and 223: the line is drawn at kDenseWords, 0.39 of the slots.
  // kept per role, a lane's share: eight bits each (a lane writes at most one
  // position of each of its warp's words, 41 of them where keys are held), in
  // streaming mode (257) 16 bits each, roles 0 .. 3 and 4 .. 7
  uint64_t kr_lo = 0, kr_hi = 0;
  const uint8_t* rp = after_wait(v.rp);
  auto put = [&](int pos, int t) {
    const uint32_t role = count_roles ? ld_u8(rp + t) : 0u;
    if (in_bounds(pos, 1, width, a.status)) dst[pos] = t;   // (the unit's own row)
    if (count_roles) {
      if constexpr (STREAM) {
        kr_lo += shl64(1ull, 16u * role);
        kr_hi += shl64(1ull, 16u * (role ^ 4u));
      } else {
        kr_lo += shl64(1ull, 8u * role);
      }
    }
  };
  {
    const int wseg = (nwords + NW - 1) / NW;
    const int q_end = min(nwords, (warp + 1) * wseg);
    int pos0 = base0 + warp_sum(lane < warp ? S.warp_tot[lane] : 0);
    for (int q0 = warp * wseg; q0 < q_end; q0 += 32) {
      const uint32_t mine = q0 + lane < q_end ? bits[q0 + lane] : 0u;
      int incl = __popc(mine);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
      }
      const int tot = __shfl_sync(0xffffffffu, incl, 31);
      if (tot > kDenseWords) {
        const uint32_t below = (1u << lane) - 1u;
#pragma unroll 8
        for (int w = 0; w < 32; ++w) {
          const uint32_t m = __shfl_sync(0xffffffffu, mine, w);
          const int first = pos0 + __shfl_sync(0xffffffffu, incl, w) - __popc(m);
          if ((m >> lane) & 1u) put(first + __popc(m & below), slot0 + (q0 + w) * 32 + lane - off);
        }
        pos0 += tot;
        continue;
      }
      for (int j0 = 0; j0 < tot; j0 += 32) {
        const int j = min(j0 + lane, tot - 1);
        int w = 0;                                 // first word with more than j bits up to it
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          if (__shfl_sync(0xffffffffu, incl, w + o - 1) <= j) w += o;
        uint32_t m = __shfl_sync(0xffffffffu, mine, w);
        int r = j - (__shfl_sync(0xffffffffu, incl, w) - __popc(m));
        int bit = 0;                               // position of the word's r-th set bit
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const int low = __popc(m & ((1u << o) - 1u));
          if (r >= low) {
            r -= low;
            m >>= o;
            bit += o;
          }
        }
        if (j0 + lane < tot) put(pos0 + j, slot0 + (q0 + w) * 32 + bit - off);
      }
      pos0 += tot;
    }
  }
  for (int64_t j = total + rank * NT + tid; j < width; j += NT * ranks) dst[j] = -1;

  if (a.keep_mask != nullptr) {
    uint8_t* mp = a.keep_mask + sbase;
    const bool mvec = ((reinterpret_cast<uintptr_t>(mp) - static_cast<uintptr_t>(off)) & 3u) == 0;
    for (int lg = tid; lg < ng; lg += NT) {
      const uint32_t m4 = (bits[lg >> 3] >> (4 * (lg & 7))) & 15u;
      const int s0 = 4 * (g0 + lg) - off;
      if (mvec && s0 >= 0 && s0 + 4 <= n) {
        const uint32_t w = (m4 & 1u) | ((m4 >> 1) & 1u) << 8 | ((m4 >> 2) & 1u) << 16 | ((m4 >> 3) & 1u) << 24;
        *reinterpret_cast<uint32_t*>(mp + s0) = w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (s0 + j >= 0 && s0 + j < n) mp[s0 + j] = static_cast<uint8_t>((m4 >> j) & 1u);
      }
    }
  }

  if (count_roles) {
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const uint32_t mine = STREAM ? static_cast<uint32_t>((r < 4 ? kr_lo : kr_hi) >> (16 * (r & 3))) & 0xFFFFu
                                   : static_cast<uint32_t>(kr_lo >> (8 * r)) & 0xFFu;
      const int c = static_cast<int>(__reduce_add_sync(0xffffffffu, mine));
      if (lane == 0 && c) {
        if constexpr (CL)
          add_rank(map_rank(&S.kept_role[r], 0), c);
        else
          atomicAdd(&S.kept_role[r], c);
      }
    }
  }
  // (no rank leaves while another may still read or add to its memory)
  unit_sync<CL>();
  if (rank == 0 && a.kept_per_role != nullptr && tid < a.n_roles)
    a.kept_per_role[static_cast<int64_t>(u) * a.n_roles + tid] =
        count_roles ? S.kept_role[tid] : S.quota[tid] + S.floor_role[tid];
  if (tid == 0 && S.nan_seen && a.status != nullptr) atomicOr(a.status, ROLEKV_STATUS_NONFINITE);
}

// Dynamic shared memory a launch may ask for: the same for every call, since
// the limit belongs to the kernel and another thread's call may set it between
// this one's setting and its launch.
constexpr int kMaxDynamicSmem = 227 * 1024 - 5 * 1024;
static_assert(sizeof(SelShared) <= 5 * 1024, "beside the dynamic part");

template <int NT, int MODE>
cudaError_t launch_select_nt(const SelectArgs& a, const SelectPlan& p, size_t smem, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(select_kernel<NT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kMaxDynamicSmem);
  if (e != cudaSuccess) return e;
  return launch_early(select_kernel<NT, MODE>, static_cast<unsigned>(a.n_units) * p.ranks, NT, smem, stream,
                      static_cast<unsigned>(p.ranks), a, p);
}

// Clusters of the plan that the device (or the partition of it that this
// context has) holds at once; alone: with at most one CTA on an SM.
template <int NT>
int64_t resident_clusters(const SelectPlan& p, size_t smem, bool alone) {
  constexpr size_t kOverHalf = 120 * 1024;         // of an SM's shared memory
  if (alone && smem < kOverHalf) smem = kOverHalf;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(p.ranks));
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = static_cast<unsigned>(p.ranks);
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int held = 0;
  if (cudaFuncSetAttribute(select_kernel<NT, kCluster>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           kMaxDynamicSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&held, select_kernel<NT, kCluster>, &cfg) != cudaSuccess) {
    cudaGetLastError();                            // (the other routes decide whether the call fails)
    return 0;
  }
  return held;
}

void plan_select(const SelectArgs& a, const SelectRoute& r, SelectPlan* p, size_t* smem) {
  const bool stream = r.mode == kStream, wide = r.wide;
  const int slots = r.groups * 4;                  // of one rank
  p->ranks = r.ranks;
  p->groups = r.groups;
  p->nb = wide ? 11 : 10;
  p->n_hist = a.policy == ROLEKV_POLICY_GLOBAL ? 1 : a.n_roles;
  p->list_cap = wide ? 8192 : slots < 4096 ? slots : 4096;
  p->hist_ints = 2 * p->n_hist * 256;
  if ((r.ranks > 1 || a.policy == ROLEKV_POLICY_SLACK) && p->hist_ints < (1 << p->nb)) p->hist_ints = 1 << p->nb;
  p->region_words = p->n_hist << (stream ? p->nb : p->nb - 1);
  const int list_words = stream ? 2 * p->list_cap : p->list_cap;
  if (p->region_words < list_words) p->region_words = list_words;
  // (16-byte aligned: groups is a multiple of 32)
  p->hist_off = (stream ? 0 : p->groups * 16) + p->groups / 8 * 4;
  *smem = static_cast<size_t>(p->hist_off) + static_cast<size_t>(p->hist_ints) * 4 +
          static_cast<size_t>(p->region_words) * 4;
}

}  // namespace

cudaError_t launch_select(const SelectArgs& a, cudaStream_t stream) {
  if (a.n_units == 0) return cudaSuccess;
  SelectPlan p;
  size_t smem;
  const SelectRoute r = select_route(a.n_max, a.n_units, device_sms(), [&](const SelectRoute& x, bool alone) {
    plan_select(a, x, &p, &smem);
    return x.threads == 1024 ? resident_clusters<1024>(p, smem, alone) : resident_clusters<512>(p, smem, alone);
  });
  plan_select(a, r, &p, &smem);
  if (r.mode == kStream) return launch_select_nt<1024, kStream>(a, p, smem, stream);
  if (r.mode == kCluster)
    return r.threads == 1024 ? launch_select_nt<1024, kCluster>(a, p, smem, stream)
                             : launch_select_nt<512, kCluster>(a, p, smem, stream);
  if (r.threads == 1024) return launch_select_nt<1024, kOne>(a, p, smem, stream);
  if (r.threads == 512) return launch_select_nt<512, kOne>(a, p, smem, stream);
  return launch_select_nt<256, kOne>(a, p, smem, stream);
}

}  // namespace rolekv
