// Dual criteria, key set and selection for ONE request, worked by a group of 256 threads
// (Eq. 9, Eq. 10; Sec. 3.3 key set).  Included by the stand-alone select kernel (one CTA per
// request) and by the single-launch filter kernel (the first eight warps of every CTA of the
// request).
//
// The per-token score is computed in fp32 with one rounding per operation (the quotients are correctly
// rounded: corrected reciprocal products where that is exact, IEEE division elsewhere), because it decides
// which indices are kept.  Budget mode is a
// radix select over the order-preserving integer image of the score, followed by an
// index-ordered emit, so kept indices come out ascending and equal scores resolve to the
// lower index.
//
// What bounds it: latency - it moves a few KB, and every barrier and shared-memory round trip is a
// serial step, and so is every instruction executed for the first time: it runs once per launch,
// from a cold instruction cache.  Hence: tokens are dealt out in strips (token j = 256 c + thread)
// and live in shared memory; the loops over the strips are real loops - one strip a trip up to 1024
// tokens, where the size of the code counts, four strips a trip (their loads overlap) beyond; a
// digit's bins are scanned by every warp for itself (no barrier), and once the cut bin holds at
// most 64 tokens - nearly always after one digit or two - they are ranked against each other directly;
// the kept set is a bitmap whose words are ballots, so positions come from popcounts.  From the
// last barrier before it to the list, in the filter kernel: 4.5 us for 576 tokens, 7.4 for 1369, 11.8 for 2880 (with
// up to 16 consecutive tokens in each thread's registers 4.6, 6.7 and 14.1).
#pragma once

#include "mustdrop_internal.h"

namespace mustdrop {

constexpr int kSelThreads = 256;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kMaxWords = kMaxVis / 32;         // words of a token bitmap
constexpr int kSelBins = 256;                   // radix digits of 8 bits
constexpr int kMaxRanked = 64;                  // tokens that are ranked against each other, one per thread
constexpr int kFewTokens = 4 * kSelThreads;     // up to here the loops over the strips take one strip a trip, else four

struct SelectParams {
  const float* g;
  const float* i;
  const int32_t* key_idx;
  const int32_t* key_cnt;
  int32_t* kept_idx;
  int32_t* kept_cnt;
  float* s_out;
  void* workspace;
  int32_t M, key_max, mode, criteria, budget, cap;
  float gamma, alpha;
  // a layer in a chain of pruning layers (all nullable): per-request token counts, original ids
  // in and out, and the key tokens' positions among the kept tokens
  const int32_t* vis_cnt;
  const int32_t* orig_in;
  int32_t* orig_out;
  int32_t* key_idx_out;
  int32_t* key_cnt_out;
  int32_t vis_start, N;                   // this request's sequence length = vis_start + its tokens + N
  int32_t gamma_default, alpha_default;   // 1: gamma = 1 / (the request's tokens), alpha = 2 / (its length)
};

// Shared state of a selection.  The bitmap, the bins and the count are cleared - and the key set
// marked - before the scores exist.
struct alignas(16) SelectShared {
  uint32_t key[kMaxWords];     // key-set bitmap (read 16 bytes at a time, as are hist and keep)
  int hist[kSelBins];
  double dsum[kSelWarps];
  uint32_t band[kSelWarps], bor[kSelWarps];   // per warp: AND / OR of the tokens' ordered score bits
  int n_ranked;
};
// Scratch that nothing has to be in before the scores are complete.
struct alignas(16) SelectScratch {
  uint32_t keep[kMaxWords];    // kept tokens
  uint32_t ties[kMaxWords];    // tokens equal to the cut, where there are too many to rank
  uint2 ranked[kMaxRanked];    // the cut bin: (ordered score bits, token)
};
__host__ __device__ constexpr int select_pad(int M) { return (M + kSelThreads - 1) / kSelThreads * kSelThreads; }

// How the 256 threads of a group meet: the whole CTA, or named barrier 1 when the group is a
// part of a larger CTA.
struct SelectSyncCta {
  static __device__ __forceinline__ void sync() { __syncthreads(); }
};
struct SelectSyncGroup {
  // (bar.sync is aligned: every lane of the warp together)
  static __device__ __forceinline__ void sync() {
    __syncwarp();
    asm volatile("bar.sync 1, 256;" ::: "memory");
  }
};

// Larger float <=> larger unsigned image (handles negative values and -0 as well).
__device__ __forceinline__ uint32_t ordered_bits(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Correctly rounded a / y for many a and one y, r = RN(1 / y): a quotient estimate and two residual
// corrections; the last one rounds correctly because the first makes the quotient faithful and r
// is correctly rounded (P. Markstein, Computation of elementary functions on the IBM RISC
// System/6000 processor, IBM J. Res. Dev. 34, 1990).  Only for operands whose residuals cannot leave
// the normal range; the others take the IEEE operation.
__device__ __forceinline__ bool plain_size(float x) { return x >= 8.6736174e-19f && x <= 1.1529215e18f; }   // 2^-60 .. 2^60
__device__ __forceinline__ float divide_by(float a, float y, float r) {
  float q = __fmul_rn(a, r);
  q = __fmaf_rn(__fmaf_rn(-q, y, a), r, q);
  return __fmaf_rn(__fmaf_rn(-q, y, a), r, q);
}

// Inclusive prefix sum over the lanes of a warp.
__device__ __forceinline__ int lane_prefix(int v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += t;
  }
  return v;
}

// Set bits of a bitmap (kMaxWords words, four per lane); every warp calls it for itself.  Lane x
// returns the number of set bits before word 4 x + pick (pick: uniform over the warp).
__device__ __forceinline__ int bitmap_prefix(const uint32_t* words, int lane, int pick, int* total) {
  const uint4 w = *reinterpret_cast<const uint4*>(&words[4 * lane]);
  const int c0 = __popc(w.x), c1 = c0 + __popc(w.y), c2 = c1 + __popc(w.z), c3 = c2 + __popc(w.w);
  const int inc = lane_prefix(c3, lane);
  *total = __shfl_sync(0xffffffffu, inc, 31);
  return inc - c3 + (pick == 0 ? 0 : (pick == 1 ? c0 : (pick == 2 ? c1 : c2)));
}

// Clears the group's shared state (`tid` of `threads` threads); touches no global data.
__device__ __forceinline__ void select_clear(SelectShared& s, int tid, int threads) {
  for (int w = tid; w < kMaxWords; w += threads) s.key[w] = 0u;
  for (int w = tid; w < kSelBins; w += threads) s.hist[w] = 0;
  if (tid == 0) s.n_ranked = 0;
}

// Marks request b's key set (`tid` of `threads` threads; repeats set the same bit).  A barrier must
// separate it from the clear before it and from select_request behind it.
__device__ __forceinline__ void select_mark_keys(const SelectParams& p, SelectShared& s, int b, int tid, int threads, bool write_out) {
  if (p.key_max <= 0) return;
  const int M = p.vis_cnt ? clamp_vis_cnt(p.vis_cnt[b], p.M) : p.M;
  const int32_t* const idx = p.key_idx + static_cast<size_t>(b) * p.key_max;
  const int given = p.key_cnt[b], first = tid < p.key_max ? idx[tid] : -1;   // (both loads under way at once)
  const int n = given < p.key_max ? given : p.key_max;
#pragma unroll 1
  for (int t = tid; t < n; t += threads) {
    const int j = t == tid ? first : idx[t];
    if (j >= 0 && j < M) atomicOr(&s.key[j >> 5], 1u << (j & 31));
    else if (write_out) record_status(p.workspace, MUSTDROP_ERR_BAD_KEY_INDEX, b * 65536 + t);
  }
}

// Selection for request b.  `tid` is the thread's index in the group (0..255).  The key set has been
// marked in s; val_g / val_i hold the request's G and I, M words each rounded up to 256 (thread tid
// reads the entries tid, tid + 256, ... first; no barrier in between is needed where it wrote them
// itself), and the tokens' ordered score bits take G's place.  With write_out the group stores
// kept_idx / kept_cnt / s_out; kept_list / kept_total, when not null, receive the same list and
// count (shared memory of the caller).
template <int kStrips, class Sync>
__device__ __forceinline__ void select_request(const SelectParams& p, SelectShared& s, SelectScratch& x, uint32_t* val_g,
                                               const uint32_t* val_i, int b, int tid, bool write_out, int32_t* kept_list,
                                               int32_t* kept_total) {
  static_assert(kSelThreads == 256 && kMaxWords <= kSelThreads && kSelBins == kSelThreads, "one thread per bin and bitmap word");
  const int lane = tid & 31, warp = tid >> 5;
  const int ld = p.M;                                    // row length of g / i / s_out / orig_in
  const int M = p.vis_cnt ? clamp_vis_cnt(p.vis_cnt[b], p.M) : p.M;   // this request's tokens
  const int n_strip = (M + kSelThreads - 1) / kSelThreads;
  float gamma = p.gamma, alpha = p.alpha;
  if (p.vis_cnt != nullptr) {                            // thresholds that default follow the request's own sizes
    if (p.gamma_default) gamma = __fdiv_rn(1.0f, static_cast<float>(M));
    if (p.alpha_default) alpha = __fdiv_rn(2.0f, static_cast<float>(p.vis_start + M + p.N));
  }
  if (tid < kMaxWords) x.keep[tid] = 0u;

  // T = sum_j g[j] in double: per thread, then fixed shuffle trees over the lanes and over the warps
  double part = 0.0;
#pragma unroll 1
  for (int c = 0; c < n_strip; c += kStrips) {
    float g[kStrips];
#pragma unroll
    for (int e = 0; e < kStrips; ++e) {
      const int j = (c + e) * kSelThreads + tid;
      g[e] = j < M ? __uint_as_float(val_g[j]) : 0.0f;
    }
#pragma unroll
    for (int e = 0; e < kStrips; ++e) part += static_cast<double>(g[e]);
  }
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) part += __shfl_xor_sync(0xffffffffu, part, d);
  if (lane == 0) s.dsum[warp] = part;
  Sync::sync();
  double tsum = s.dsum[lane & (kSelWarps - 1)];
#pragma unroll
  for (int d = kSelWarps / 2; d >= 1; d >>= 1) tsum += __shfl_xor_sync(0xffffffffu, tsum, d);
  const float gt = __fmul_rn(gamma, static_cast<float>(tsum));

  // Scores of the thread's tokens, as ordered integers (threshold mode: 1 = the rule keeps the
  // token).  Bits that all of the request's scores share need no radix pass (scores of one request
  // lie within a few powers of two: their top bits are the same for all, and a pass over them would
  // be every thread's atomics on one or two counters): AND and OR over the tokens, per warp here,
  // over the group behind the barrier below.
  const bool threshold = p.mode == MUSTDROP_MODE_THRESHOLD;
  const bool use_g = p.criteria != MUSTDROP_CRIT_INDIVIDUAL_ONLY, use_i = p.criteria != MUSTDROP_CRIT_GLOBAL_ONLY;
  const bool plain = plain_size(gt) && plain_size(alpha);
  const float r_gt = __frcp_rn(gt), r_alpha = __frcp_rn(alpha);
  float* const s_row = write_out && p.s_out != nullptr ? p.s_out + static_cast<size_t>(b) * ld : nullptr;
  uint32_t all_and = 0xffffffffu, all_or = 0u;
#pragma unroll 1
  for (int c = 0; c < n_strip; c += kStrips) {
    float g[kStrips], i[kStrips], gs[kStrips], is[kStrips];
    bool quick = plain;
#pragma unroll
    for (int e = 0; e < kStrips; ++e) {
      const int j = (c + e) * kSelThreads + tid, at = j < M ? j : tid;
      g[e] = __uint_as_float(val_g[at]);
      i[e] = __uint_as_float(val_i[at]);
    }
#pragma unroll
    for (int e = 0; e < kStrips; ++e) {
      quick = quick && plain_size(g[e]) && plain_size(i[e]);
      gs[e] = divide_by(g[e], gt, r_gt);
      is[e] = divide_by(i[e], alpha, r_alpha);
    }
    if (!quick) {
#pragma unroll 1
      for (int e = 0; e < kStrips; ++e) {   // (a rotation keeps the arrays in registers without copies of the divisions)
        const float g0 = g[0], i0 = i[0];
#pragma unroll
        for (int k = 0; k + 1 < kStrips; ++k) { g[k] = g[k + 1]; i[k] = i[k + 1]; gs[k] = gs[k + 1]; is[k] = is[k + 1]; }
        g[kStrips - 1] = g0; i[kStrips - 1] = i0;
        gs[kStrips - 1] = __fdiv_rn(g0, gt); is[kStrips - 1] = __fdiv_rn(i0, alpha);
      }
    }
#pragma unroll
    for (int e = 0; e < kStrips; ++e) {
      const int j = (c + e) * kSelThreads + tid;
      const float sc = !use_i || (use_g && gs[e] > is[e]) ? gs[e] : is[e];
      const bool drop = (!use_g || g[e] <= gt) && (!use_i || i[e] < alpha);   // Eq. 9, Eq. 10
      const uint32_t u = threshold ? (drop ? 0u : 1u) : ordered_bits(sc);
      if (j < M) {
        val_g[j] = u;
        all_and &= u;
        all_or |= u;
        if (s_row != nullptr) s_row[j] = sc;
      }
    }
  }
  all_and = __reduce_and_sync(0xffffffffu, all_and);
  all_or = __reduce_or_sync(0xffffffffu, all_or);
  if (lane == 0) {
    s.band[warp] = all_and;
    s.bor[warp] = all_or;
  }
  Sync::sync();

  // Which candidates (tokens outside the key set) are kept: those with (u & mask) > prefix, and of
  // those with (u & mask) == prefix all (kAll), none (kNone), or the `remaining` best - ranked
  // directly (kRank), or the lowest indices among full ties (kTies).
  enum { kNone, kAll, kRank, kTies };
  uint32_t prefix = 0u, mask = 0xffffffffu;   // (threshold mode: keep what is above 0)
  int equal = kNone, remaining = 0;
  if (!threshold) {
    int n_key;
    (void)bitmap_prefix(s.key, lane, 0, &n_key);
    const int want = p.budget - n_key;
    if (want <= 0) {
      prefix = 0xffffffffu;                              // (nothing is above it)
    } else if (want >= M - n_key) {
      mask = 0u;                                         // every candidate equals the empty prefix
      equal = kAll;
    } else {
      // radix select of the want-th largest candidate: digits of eight bits from the highest bit in
      // which two tokens differ downwards (the bits above it are the same in every candidate)
      const uint32_t g_and = __reduce_and_sync(0xffffffffu, s.band[lane & (kSelWarps - 1)]);
      const uint32_t g_or = __reduce_or_sync(0xffffffffu, s.bor[lane & (kSelWarps - 1)]);
      const uint32_t differ = g_and ^ g_or;
      const int hb = differ ? 31 - __clz(differ) : 7;                  // (all equal: one pass over the low bits)
      mask = hb >= 31 ? 0u : ~((2u << hb) - 1u);                        // the shared bits
      prefix = g_and & mask;
      remaining = want;
#pragma unroll 1
      for (int shift = hb >= 7 ? hb - 7 : 0;; shift = shift > 8 ? shift - 8 : 0) {
#pragma unroll 1
        for (int c = 0; c < n_strip; c += kStrips) {
          uint32_t u[kStrips], key[kStrips];
#pragma unroll
          for (int e = 0; e < kStrips; ++e) {
            const int j = (c + e) * kSelThreads + tid, at = j < M ? j : tid;
            key[e] = j < M ? s.key[at >> 5] : 0xffffffffu;
            u[e] = val_g[at];
          }
#pragma unroll
          for (int e = 0; e < kStrips; ++e)
            if (!((key[e] >> lane) & 1u) && (u[e] & mask) == prefix) atomicAdd(&s.hist[(u[e] >> shift) & (kSelBins - 1)], 1);
        }
        Sync::sync();
        // digit d is the cut iff (#candidates with a larger digit) < remaining <= that + hist[d].
        // Every warp scans the bins for itself: eight per lane, the highest in lane 0.
        constexpr int kPer = kSelBins / 32;
        int bins[kPer];   // descending digits
        const int4* const mine = reinterpret_cast<const int4*>(&s.hist[kSelBins - kPer * (lane + 1)]);
#pragma unroll
        for (int e = 0; e < kPer / 4; ++e) {
          const int4 v = mine[kPer / 4 - 1 - e];
          bins[4 * e] = v.w; bins[4 * e + 1] = v.z; bins[4 * e + 2] = v.y; bins[4 * e + 3] = v.x;
        }
        int sum = 0;
#pragma unroll
        for (int e = 0; e < kPer; ++e) sum += bins[e];
        int above = lane_prefix(sum, lane) - sum;
        int digit = -1, left = 0, here = 0;
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
          if (above < remaining && remaining <= above + bins[e]) {
            digit = kSelBins - kPer * lane - 1 - e;
            left = remaining - above;
            here = bins[e];
          }
          above += bins[e];
        }
        const int owner = __ffs(__ballot_sync(0xffffffffu, digit >= 0)) - 1;
        digit = __shfl_sync(0xffffffffu, digit, owner);
        remaining = __shfl_sync(0xffffffffu, left, owner);
        here = __shfl_sync(0xffffffffu, here, owner);
        // (the lowest digit may reach over bits that are resolved already: they are the same in
        // every token still in the running, so the bins keep their order)
        const uint32_t field = static_cast<uint32_t>(kSelBins - 1) << shift;
        prefix = (prefix & ~field) | (static_cast<uint32_t>(digit) << shift);
        mask |= field;
        if (remaining == here) { equal = kAll; break; }     // the whole bin is taken: lower digits cannot matter
        if (here <= kMaxRanked) { equal = kRank; break; }
        if (shift == 0) { equal = kTies; break; }
        Sync::sync();                                        // every warp has read the histogram
        s.hist[tid] = 0;
        Sync::sync();
      }
    }
  }

  // the kept set as a bitmap: one ballot per strip and warp
#pragma unroll 1
  for (int c = 0; c < n_strip; c += kStrips) {
    uint32_t u[kStrips], key[kStrips], same[kStrips];
    int base[kStrips];
#pragma unroll
    for (int e = 0; e < kStrips; ++e) {
      const int j = (c + e) * kSelThreads + tid, w = (c + e) * kSelWarps + warp;
      key[e] = w < kMaxWords ? s.key[w] : 0u;
      u[e] = val_g[j < M ? j : tid];
    }
#pragma unroll
    for (int e = 0; e < kStrips; ++e) {
      const int j = (c + e) * kSelThreads + tid, w = (c + e) * kSelWarps + warp;
      const bool cand = j < M && !((key[e] >> lane) & 1u);
      same[e] = __ballot_sync(0xffffffffu, cand && (u[e] & mask) == prefix);
      const uint32_t over = __ballot_sync(0xffffffffu, cand && (u[e] & mask) > prefix);
      base[e] = 0;
      if (lane == 0 && w < kMaxWords) {
        x.keep[w] = over | key[e] | (equal == kAll ? same[e] : 0u);
        if (equal == kTies) x.ties[w] = same[e];
        if (equal == kRank && same[e] != 0u) base[e] = atomicAdd(&s.n_ranked, __popc(same[e]));
      }
    }
    if (equal == kRank) {   // (uniform over the group)
#pragma unroll
      for (int e = 0; e < kStrips; ++e) {
        const int at = __shfl_sync(0xffffffffu, base[e], 0) + __popc(same[e] & ((1u << lane) - 1u));
        if ((same[e] >> lane) & 1u) x.ranked[at] = make_uint2(u[e], static_cast<uint32_t>((c + e) * kSelThreads + tid));
      }
    }
  }
  Sync::sync();
  if (equal >= kRank) {   // uniform over the group
    if (equal == kRank) {
      const int n = s.n_ranked;
      if (tid < n) {
        const uint2 me = x.ranked[tid];
        int better = 0;
#pragma unroll 4
        for (int y = 0; y < n; ++y) {
          const uint2 o = x.ranked[y];
          better += (o.x > me.x || (o.x == me.x && o.y < me.y)) ? 1 : 0;
        }
        if (better < remaining) atomicOr(&x.keep[me.y >> 5], 1u << (me.y & 31u));
      }
    } else if (tid < n_strip * kSelWarps) {
      int before = 0;
#pragma unroll 1
      for (int y = 0; y < tid; ++y) before += __popc(x.ties[y]);
      uint32_t rest = x.ties[tid], take = 0u;
#pragma unroll 1
      for (int n = remaining - before; n > 0 && rest != 0u; --n) {
        take |= rest & (0u - rest);
        rest &= rest - 1u;
      }
      x.keep[tid] |= take;
    }
    Sync::sync();
  }

  // index-ordered emit
  int total, key_total = 0, key_before = 0;
  const int before = bitmap_prefix(x.keep, lane, warp & 3, &total);
  // a chain of layers also wants the kept tokens' original ids and where the key tokens went
  const bool emit_keys = write_out && p.key_idx_out != nullptr && p.key_max > 0;   // uniform over the group
  if (emit_keys) key_before = bitmap_prefix(s.key, lane, warp & 3, &key_total);
#pragma unroll 1
  for (int c = 0; c < n_strip; c += kStrips) {
    uint32_t keep[kStrips];
    int pos[kStrips];
    const uint32_t below = (1u << lane) - 1u;
#pragma unroll
    for (int e = 0; e < kStrips; ++e) {
      const int w = (c + e) * kSelWarps + warp;
      keep[e] = w < kMaxWords ? x.keep[w] : 0u;
      pos[e] = __shfl_sync(0xffffffffu, before, (w >> 2) & 31) + __popc(keep[e] & below);
    }
#pragma unroll
    for (int e = 0; e < kStrips; ++e) {
      const int j = (c + e) * kSelThreads + tid;
      if (((keep[e] >> lane) & 1u) && pos[e] < p.cap) {
        if (kept_list != nullptr) kept_list[pos[e]] = j;
        if (write_out) {
          p.kept_idx[static_cast<size_t>(b) * p.cap + pos[e]] = j;
          if (p.orig_out != nullptr)
            p.orig_out[static_cast<size_t>(b) * p.cap + pos[e]] =
                p.orig_in != nullptr ? p.orig_in[static_cast<size_t>(b) * ld + j] : j;
        }
      }
      if (emit_keys) {
        const int w = (c + e) * kSelWarps + warp;
        const uint32_t key = w < kMaxWords ? s.key[w] : 0u;
        const int key_pos = __shfl_sync(0xffffffffu, key_before, (w >> 2) & 31) + __popc(key & below);
        if (((key >> lane) & 1u) && pos[e] < p.cap && key_pos < p.key_max)
          p.key_idx_out[static_cast<size_t>(b) * p.key_max + key_pos] = pos[e];
      }
    }
  }
  if (tid == 0) {
    if (write_out) {
      p.kept_cnt[b] = total;
      if (p.key_cnt_out != nullptr) p.key_cnt_out[b] = emit_keys ? (key_total < p.key_max ? key_total : p.key_max) : 0;
    }
    if (kept_total != nullptr) *kept_total = total;
  }
}

}  // namespace mustdrop
