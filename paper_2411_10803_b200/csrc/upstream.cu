// Vision-encoding stage of the method (Sec. 3.3), upstream of the prefill filter:
//   Local Spatial Merging (Eq. 5): non-overlapping 2 x 2 windows of the token grid whose mean
//     pairwise cosine similarity exceeds tau collapse into one averaged token at the window's
//     first slot; the survivors are packed in raster order;
//   Key Retaining (Eq. 6-7): head-averaged [CLS] attention over the patch tokens, and the tokens
//     above an adaptive threshold form the key set O.  The paper names no threshold rule; here it
//     is Tukey's upper fence Q3 + 1.5 (Q3 - Q1) with linearly interpolated quartiles.
// A thread-block cluster of up to eight CTAs of 256 threads works on one image (windows, rows and
// tokens are dealt out over the cluster's CTAs; flags, softmax statistics and attention cross through
// distributed shared memory, in a fixed order).  Bound: reading the input once (1.2 MB per image at
// 576 tokens x 1024 channels, the merge also writes ~0.9 MB), and the serial steps between the
// cluster's barriers, which all images of a batch reach at about the same time.
#include <cuda_bf16.h>

#include <atomic>

#include "mustdrop_internal.h"
#include "vision_plan.h"

namespace mustdrop {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
static_assert(kWarps == kVisionWarps, "the layout rules count the warps of a CTA");
constexpr int kMaxSlots = 4096;            // tokens per image
constexpr int kWords = kMaxSlots / 32;     // words of a token bitmap

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  __syncwarp();   // (.aligned: every lane of the warp together)
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The two halves of the barrier.  Shared memory of another CTA may only be touched once that CTA
// is known to have started: every kernel arrives in its prologue and waits before its first
// remote store, so the wait costs nothing unless a peer really is late.
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of a shared-memory object of this CTA, as seen in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_addr(const void* local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(r)
               : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(local))), "r"(rank));
  return r;
}

// Set bits of a bitmap of kWords words before each of the four words 4 lane .. 4 lane + 3; every
// warp calls it for itself.
__device__ __forceinline__ void bitmap_prefix(const uint32_t* words, int lane, int (&before)[4], int* total) {
  const uint4 w = *reinterpret_cast<const uint4*>(&words[4 * lane]);
  const int c0 = __popc(w.x), c1 = c0 + __popc(w.y), c2 = c1 + __popc(w.z), c3 = c2 + __popc(w.w);
  int inc = c3;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= d) inc += t;
  }
  *total = __shfl_sync(0xffffffffu, inc, 31);
  before[0] = inc - c3;
  before[1] = before[0] + c0;
  before[2] = before[0] + c1;
  before[3] = before[0] + c2;
}

// Two fp32 operations per instruction.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float sum2(uint64_t v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return lo + hi;
}

// ---- Local Spatial Merging ----------------------------------------------------------------------
struct MergeParams {
  const uint4* tokens;   // [B, g*g, C/8]
  uint4* merged;         // [B, g*g, C/8]
  int32_t* slots;        // [B, g*g]
  int32_t* merged_cnt;   // [B]
  float* window_sim;     // [B, (g/2)^2] or null
  int32_t grid, vecs;    // vecs = C / 8
  uint32_t inv_grid, inv_half;   // ceil(2^20 / grid), ceil(2^20 / (grid / 2)): exact quotients of numbers below 4096
  float tau;
};

__device__ __forceinline__ int quotient(int x, uint32_t inv) { return static_cast<int>((static_cast<uint32_t>(x) * inv) >> 20); }

// FLY: vectors of each of a window's four tokens that a lane has in flight.  Two take the registers of a fourth CTA on
// the SM, which rows of 32 vectors or fewer would give away for nothing.
template <int FLY>
__global__ void __launch_bounds__(kThreads, FLY == 2 ? 3 : 4) spatial_merge_kernel(MergeParams p) {
  __shared__ unsigned char merged_flag[kMaxSlots / 4];
  __shared__ __align__(16) uint32_t emit[kWords];   // slots that emit a token: all of an unmerged window, the first of a merged one
  __shared__ int first_row[kWords];                 // output row of a word's first emitting slot
  const int C = static_cast<int>(cluster_size()), rank = static_cast<int>(cluster_rank());
  const int b = blockIdx.x / C, g = p.grid, gw = g / 2, n_win = gw * gw, n_slot = g * g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  cluster_arrive();          // "this CTA runs": peers wait for it before their first remote store
  bool peers_started = false;
  for (int w = threadIdx.x; w < kWords; w += kThreads) emit[w] = 0u;
  pdl_launch_dependents();
  pdl_wait();
  const uint4* in = p.tokens + static_cast<size_t>(b) * n_slot * p.vecs;

  // 1. per window: the four norms and six dot products, fp32 accumulation, two channels per
  //    instruction.  The cluster's warps share the windows; a window's flag is stored into every
  //    CTA's copy of the flag array.
  for (int w = rank * kWarps + warp; w < n_win; w += C * kWarps) {
    const int wy = quotient(w, p.inv_half), wx = w - wy * gw;
    const uint4* r0 = in + static_cast<size_t>(2 * wy * g + 2 * wx) * p.vecs;
    const uint4* r1 = r0 + p.vecs;                          // (y, x+1)
    const uint4* r2 = r0 + static_cast<size_t>(g) * p.vecs; // (y+1, x)
    const uint4* r3 = r2 + p.vecs;
    uint64_t acc[10] = {};   // |0|^2 |1|^2 |2|^2 |3|^2 01 | 02 03 12 13 23
#pragma unroll 1
    for (int x = lane; x < p.vecs; x += 32 * FLY) {
      uint4 t[FLY][4];
#pragma unroll
      for (int u = 0; u < FLY; ++u) {
        const int at = x + 32 * u;
        const bool in = at < p.vecs;
        t[u][0] = in ? r0[at] : make_uint4(0, 0, 0, 0);
        t[u][1] = in ? r1[at] : make_uint4(0, 0, 0, 0);
        t[u][2] = in ? r2[at] : make_uint4(0, 0, 0, 0);
        t[u][3] = in ? r3[at] : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < FLY; ++u) {
        const uint32_t aw[4] = {t[u][0].x, t[u][0].y, t[u][0].z, t[u][0].w}, cw[4] = {t[u][1].x, t[u][1].y, t[u][1].z, t[u][1].w};
        const uint32_t ew[4] = {t[u][2].x, t[u][2].y, t[u][2].z, t[u][2].w}, fw[4] = {t[u][3].x, t[u][3].y, t[u][3].z, t[u][3].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint64_t v0 = pack2(bf16_lo(aw[q]), bf16_hi(aw[q])), v1 = pack2(bf16_lo(cw[q]), bf16_hi(cw[q]));
          const uint64_t v2 = pack2(bf16_lo(ew[q]), bf16_hi(ew[q])), v3 = pack2(bf16_lo(fw[q]), bf16_hi(fw[q]));
          fma2(acc[0], v0, v0); fma2(acc[1], v1, v1); fma2(acc[2], v2, v2); fma2(acc[3], v3, v3);
          fma2(acc[4], v0, v1); fma2(acc[5], v0, v2); fma2(acc[6], v0, v3);
          fma2(acc[7], v1, v2); fma2(acc[8], v1, v3); fma2(acc[9], v2, v3);
        }
      }
    }
    // sums over the lanes: the half-warps exchange five sums for five, then each reduces its own five
    const bool upper = lane >= 16;
    float v[5], o[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const float lo = sum2(acc[i]), hi = sum2(acc[i + 5]);
      v[i] = (upper ? hi : lo) + __shfl_xor_sync(0xffffffffu, upper ? lo : hi, 16);
    }
#pragma unroll
    for (int d = 8; d >= 1; d >>= 1)
#pragma unroll
      for (int i = 0; i < 5; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], d);
#pragma unroll
    for (int i = 0; i < 5; ++i) o[i] = __shfl_xor_sync(0xffffffffu, v[i], 16);   // (lower lanes: the upper ones' sums)
    if (!peers_started) {   // (warp-uniform) every CTA of the cluster has started: its shared memory exists
      cluster_wait();
      peers_started = true;
    }
    const float tiny = 1e-30f;
    const float l0 = fmaxf(sqrtf(v[0]), tiny), l1 = fmaxf(sqrtf(v[1]), tiny), l2 = fmaxf(sqrtf(v[2]), tiny), l3 = fmaxf(sqrtf(v[3]), tiny);
    const float sim = (v[4] / (l0 * l1) + o[0] / (l0 * l2) + o[1] / (l0 * l3) + o[2] / (l1 * l2) + o[3] / (l1 * l3) +
                       o[4] / (l2 * l3)) * (1.0f / 6.0f);   // (lane 0's is the one that counts)
    const uint32_t flag = __shfl_sync(0xffffffffu, sim > p.tau ? 1u : 0u, 0);
    if (lane < C)
      asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(peer_addr(&merged_flag[w], lane)), "r"(flag) : "memory");
    if (lane == 0 && p.window_sim != nullptr) p.window_sim[static_cast<size_t>(b) * n_win + w] = sim;
  }
  if (!peers_started) cluster_wait();   // a warp without a window: complete the prologue's barrier
  cluster_barrier();   // every flag has arrived in every CTA; no remote store after this point

  // 2. which slots emit a token and where: a bitmap in raster order and its prefix counts, by every
  //    CTA for itself
  const int n_word = (n_slot + 31) / 32;
  for (int w = warp; w < n_word; w += kWarps) {
    const int s = 32 * w + lane, y = quotient(s, p.inv_grid), x = s - y * g;
    const bool m = s < n_slot && merged_flag[(y >> 1) * gw + (x >> 1)] != 0;
    const uint32_t word = __ballot_sync(0xffffffffu, s < n_slot && (!m || ((y | x) & 1) == 0));
    if (lane == 0) emit[w] = word;
  }
  __syncthreads();
  if (warp == 0) {
    int before[4], total;
    bitmap_prefix(emit, lane, before, &total);
    *reinterpret_cast<int4*>(&first_row[4 * lane]) = make_int4(before[0], before[1], before[2], before[3]);
    if (lane == 0 && rank == 0) p.merged_cnt[b] = total;
  }
  __syncthreads();
  auto row_of = [&](int s) { return first_row[s >> 5] + __popc(emit[s >> 5] & ((1u << (s & 31)) - 1u)); };
  for (int w = rank * kWarps + warp; w < n_word; w += C * kWarps)
    if ((emit[w] >> lane) & 1u) p.slots[static_cast<size_t>(b) * n_slot + row_of(32 * w + lane)] = 32 * w + lane;

  // 3. the surviving rows: copies of the tokens of unmerged windows, two rows and eight 16-byte loads
  //    per lane in flight, ...  (The tokens are read a second time, from L2 as far as they are still
  //    there.  Hints that keep them - evict_last on the first reading - make this kernel 10 % faster and
  //    the key set behind it slower by more.)
  uint4* out = p.merged + static_cast<size_t>(b) * n_slot * p.vecs;
  for (int s0 = rank * kWarps + warp; s0 < n_slot; s0 += 2 * C * kWarps) {
    const uint4* src[2];
    uint4* dst[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int s = s0 + i * C * kWarps, y = quotient(s, p.inv_grid), x = s - y * g;
      const bool copy = s < n_slot && merged_flag[(y >> 1) * gw + (x >> 1)] == 0;
      src[i] = copy ? in + static_cast<size_t>(s) * p.vecs : nullptr;
      dst[i] = copy ? out + static_cast<size_t>(row_of(s)) * p.vecs : nullptr;
    }
    for (int v0 = lane; v0 < p.vecs; v0 += 4 * 32) {
      uint4 t[2][4];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (src[i] != nullptr && v0 + 32 * u < p.vecs) t[i][u] = src[i][v0 + 32 * u];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (src[i] != nullptr && v0 + 32 * u < p.vecs) __stcs(dst[i] + v0 + 32 * u, t[i][u]);
    }
  }
  //    ... and the plain average of every merged window in fp32, rounded once
  for (int w = rank * kWarps + warp; w < n_win; w += C * kWarps) {
    if (merged_flag[w] == 0) continue;
    const int wy = quotient(w, p.inv_half), wx = w - wy * gw, s = 2 * wy * g + 2 * wx;
    const uint4* r0 = in + static_cast<size_t>(s) * p.vecs;
    const uint4* r1 = r0 + p.vecs;
    const uint4* r2 = r0 + static_cast<size_t>(g) * p.vecs;
    const uint4* r3 = r2 + p.vecs;
    uint4* dst = out + static_cast<size_t>(row_of(s)) * p.vecs;
#pragma unroll 1
    for (int v0 = lane; v0 < p.vecs; v0 += 32 * FLY) {
      uint4 t[FLY][4];
#pragma unroll
      for (int u = 0; u < FLY; ++u) {
        const int at = min(v0 + 32 * u, p.vecs - 1);
        t[u][0] = r0[at]; t[u][1] = r1[at]; t[u][2] = r2[at]; t[u][3] = r3[at];
      }
#pragma unroll
      for (int u = 0; u < FLY; ++u) {
        const uint32_t aw[4] = {t[u][0].x, t[u][0].y, t[u][0].z, t[u][0].w}, cw[4] = {t[u][1].x, t[u][1].y, t[u][1].z, t[u][1].w};
        const uint32_t ew[4] = {t[u][2].x, t[u][2].y, t[u][2].z, t[u][2].w}, fw[4] = {t[u][3].x, t[u][3].y, t[u][3].z, t[u][3].w};
        uint32_t ow[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float lo = ((bf16_lo(aw[q]) + bf16_lo(cw[q])) + (bf16_lo(ew[q]) + bf16_lo(fw[q]))) * 0.25f;
          const float hi = ((bf16_hi(aw[q]) + bf16_hi(cw[q])) + (bf16_hi(ew[q]) + bf16_hi(fw[q]))) * 0.25f;
          const __nv_bfloat16 bl = __float2bfloat16_rn(lo), bh = __float2bfloat16_rn(hi);
          ow[q] = static_cast<uint32_t>(__bfloat16_as_ushort(bl)) | (static_cast<uint32_t>(__bfloat16_as_ushort(bh)) << 16);
        }
        if (v0 + 32 * u < p.vecs) __stcs(dst + v0 + 32 * u, make_uint4(ow[0], ow[1], ow[2], ow[3]));
      }
    }
  }
}

// ---- Key Retaining ------------------------------------------------------------------------------
constexpr int kParts = 2;         // a head's tokens of a CTA are two warps' work: 12 or 16 heads deal out evenly
constexpr int kRanked = 64;       // tokens that are ranked against each other for a quartile, one per thread
constexpr int kHalf = kThreads / 2;   // threads that work on a quartile

struct KeySetParams {
  const __nv_bfloat16* q_cls;   // [B, H, D]
  const uint4* k;               // [B, H, M, D/8]
  float* a_cls;                 // [B, M] or null
  float* mu_out;                // [B] or null
  int32_t* key_idx;             // [B, key_max]
  int32_t* key_cnt;             // [B]
  int32_t H, D, M, key_max;
  int32_t part;                 // tokens of a warp's unit of work: ceil(ceil(M / CTAs) / kParts)
  int32_t block;                // heads whose logits fit a CTA's shared memory at a time
  float scale_log2e;
};

// The cluster's CTAs share the TOKENS: every CTA reads its share of every head's keys (all its loads
// are independent, nothing is between them), a warp at a time the logits of one head and half of the
// CTA's tokens, their maximum and the sum of their exponentials; one exchange of these statistics
// over the cluster normalises all heads.  (Sharing the heads put six CTA-wide barriers into every
// head and left the partial sums of all tokens to be exchanged: 36 us for 64 images of 576 tokens,
// 16 heads x 64, where reading the keys takes 11.5 us.)
// LANES, VPL, FLY: a token's row is read by LANES = 4 or 8 lanes, VPL vectors of 16 bytes each, and a warp takes 32 / LANES
// tokens a step, FLY steps a trip.  (A lane per vector and a power of two of lanes to a token leaves 5 to 7 of 16 lanes idle
// at 72, 80 and 88 dimensions, and takes three or four shuffles for two or four tokens instead of two for eight:
// 49 images of 1936 tokens, 16 x 80: 120.4 -> 67.7 us, 64 of 576: 45.8 -> 33.9; memory takes 37.4 and 14.5.)  LANES = 0: a
// lane per vector, VPL = 1.
// AHEAD: a trip's loads go out before the products of the trip before, which takes the registers of as many loads again.
template <int LANES, int VPL, int FLY, bool AHEAD>
__global__ void __launch_bounds__(kThreads, 4) key_set_kernel(KeySetParams p) {
  __shared__ __align__(16) float a[kMaxSlots];      // CTA 0: head-mean attention; the others: of their own tokens
  __shared__ __align__(16) uint32_t words[kWords];
  __shared__ __align__(16) int hist[2][256];        // (one set per quartile)
  __shared__ uint32_t ranked[2][kRanked], over[2];  // values of the cut bin; the smallest value above it
  __shared__ int n_ranked[2];
  __shared__ uint32_t order[2][2];                  // per quartile the two order statistics it interpolates
  __shared__ uint32_t band[kWarps], bor[kWarps];
  extern __shared__ __align__(16) unsigned char dyn[];
  const int C = static_cast<int>(cluster_size()), rank = static_cast<int>(cluster_rank());
  const int b = blockIdx.x / C, M = p.M, dv = p.D / 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* const stat = reinterpret_cast<float2*>(dyn);                  // [CTA][unit] (maximum, sum)
  float2* const norm = stat + C * p.block * kParts;                     // [head] (maximum, 1 / (H sum)) over all tokens
  float* const logits = reinterpret_cast<float*>(norm + p.block);       // [unit][part], log2 units
  cluster_arrive();          // "this CTA runs": peers wait for it before their first remote store
  bool peers_started = false;
  hist[0][threadIdx.x] = 0;
  hist[1][threadIdx.x] = 0;
  if (threadIdx.x < kWords) words[threadIdx.x] = 0u;
  if (threadIdx.x < 2) {
    n_ranked[threadIdx.x] = 0;
    over[threadIdx.x] = 0xffffffffu;
  }
  pdl_launch_dependents();
  pdl_wait();
  const float inv_h = 1.0f / static_cast<float>(p.H);
  const int own = kParts * p.part, t0 = rank * own, n_own = max(0, min(own, M - t0));   // this CTA's tokens
  int grp = LANES > 0 ? LANES : 1;                  // lanes that share a token's row
  if constexpr (LANES == 0) {
    while (grp < dv) grp <<= 1;
  }
  const int sub = lane & (grp - 1), tok = lane / grp, per_warp = 32 / grp;
  float* const mine = a + t0;                       // (at the place where CTA 0 wants them)

  for (int hb = 0; hb < p.H; hb += p.block) {
    const int nh = min(p.block, p.H - hb), units = nh * kParts;
    // A unit's trips.  With AHEAD the next trip's loads - of the next unit, behind a unit's last - go out before this one's
    // products.  (Five steps of a vector each without loads ahead: 20 us until the last logit of 64 images of 576
    // tokens, 16 heads x 64, where memory takes 11.6; the kernel 30.8 us, with loads ahead 28.5.)
    const uint4* const k_img = p.k + (static_cast<size_t>(b) * p.H + hb) * M * dv;
    auto fetch = [&](int u, int base, uint4 (&kv)[FLY][VPL]) {
      const int first = (u % kParts) * p.part, n = max(0, min(p.part, n_own - first));
      const uint4* const rows = k_img + (static_cast<size_t>(u / kParts) * M + t0 + first) * dv + sub;
#pragma unroll
      for (int x = 0; x < FLY; ++x) {
        const int j = base + x * per_warp + tok;
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          kv[x][v] = make_uint4(0, 0, 0, 0);
          if (u < units && j < n && sub + v * grp < dv) kv[x][v] = rows[static_cast<size_t>(j) * dv + v * grp];
        }
      }
    };
    uint4 kv[FLY][VPL];
    [[maybe_unused]] uint4 next[FLY][VPL];
    if constexpr (AHEAD) fetch(warp, 0, kv);
    for (int u = warp; u < units; u += kWarps) {
      const int h = hb + u / kParts, first = (u % kParts) * p.part, n = max(0, min(p.part, n_own - first));
      uint4 qw[VPL];
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        qw[v] = make_uint4(0, 0, 0, 0);
        if (sub + v * grp < dv) qw[v] = reinterpret_cast<const uint4*>(p.q_cls)[(static_cast<size_t>(b) * p.H + h) * dv + sub + v * grp];
      }
      float* const z = logits + u * p.part;
      float mx = -INFINITY;
      for (int base = 0;; base += FLY * per_warp) {   // warp-uniform trip count, at least one
        const bool last = base + FLY * per_warp >= n;
        if constexpr (AHEAD) fetch(last ? u + kWarps : u, last ? 0 : base + FLY * per_warp, next);
        else fetch(u, base, kv);
#pragma unroll
        for (int x = 0; x < FLY; ++x) {
          const int j = base + x * per_warp + tok;
          float da = 0.0f;
#pragma unroll
          for (int v = 0; v < VPL; ++v) {   // (a sum per vector: chains of eight terms, as with a lane per vector)
            float dv8 = bf16_lo(kv[x][v].x) * bf16_lo(qw[v].x);
            dv8 = fmaf(bf16_hi(kv[x][v].x), bf16_hi(qw[v].x), dv8);
            dv8 = fmaf(bf16_lo(kv[x][v].y), bf16_lo(qw[v].y), dv8);
            dv8 = fmaf(bf16_hi(kv[x][v].y), bf16_hi(qw[v].y), dv8);
            dv8 = fmaf(bf16_lo(kv[x][v].z), bf16_lo(qw[v].z), dv8);
            dv8 = fmaf(bf16_hi(kv[x][v].z), bf16_hi(qw[v].z), dv8);
            dv8 = fmaf(bf16_lo(kv[x][v].w), bf16_lo(qw[v].w), dv8);
            dv8 = fmaf(bf16_hi(kv[x][v].w), bf16_hi(qw[v].w), dv8);
            da = v == 0 ? dv8 : da + dv8;
          }
          for (int d = grp >> 1; d >= 1; d >>= 1) da += __shfl_xor_sync(0xffffffffu, da, d);   // over the group's lanes (fixed tree)
          if (j < n) {
            da *= p.scale_log2e;
            if (sub == 0) z[j] = da;
            mx = fmaxf(mx, da);
          }
        }
#pragma unroll
        for (int x = 0; x < FLY; ++x)
#pragma unroll
          for (int v = 0; v < VPL; ++v)
            if constexpr (AHEAD) kv[x][v] = next[x][v];
        if (last) break;
      }
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
      __syncwarp();
      float sum = 0.0f;
      for (int j = lane; j < n; j += 32) sum += exp2f(z[j] - mx);
      sum = warp_sum(sum);
      if (!peers_started) {   // (warp-uniform) every CTA of the cluster has started: its shared memory exists
        cluster_wait();
        peers_started = true;
      }
      if (lane < C)
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(peer_addr(&stat[rank * units + u], lane)), "f"(mx), "f"(sum)
                     : "memory");
    }
    if (!peers_started) {
      cluster_wait();
      peers_started = true;
    }
    cluster_barrier();   // every CTA's statistics of these heads are everywhere
    for (int h = threadIdx.x; h < nh; h += kThreads) {
      float m = -INFINITY, total = 0.0f;
      for (int c = 0; c < C; ++c)
        for (int x = 0; x < kParts; ++x) m = fmaxf(m, stat[c * units + h * kParts + x].x);
      for (int c = 0; c < C; ++c)
        for (int x = 0; x < kParts; ++x) {
          const float2 v = stat[c * units + h * kParts + x];
          total = fmaf(v.y, exp2f(v.x - m), total);       // (no token: (-inf, 0))
        }
      norm[h] = make_float2(m, inv_h / total);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < n_own; t += kThreads) {
      const int part = t / p.part, at = t - part * p.part;
      float sum = hb == 0 ? 0.0f : mine[t];
      for (int h = 0; h < nh; ++h)   // (from the logits: tokens with equal keys get equal bits whoever holds them)
        sum = fmaf(exp2f(logits[(h * kParts + part) * p.part + at] - norm[h].x), norm[h].y, sum);
      mine[t] = sum;
    }
    if (hb + p.block < p.H) cluster_barrier();   // the statistics are read: the next heads' may come
  }
  for (int t = threadIdx.x; t < n_own; t += kThreads) {   // (each thread its own sums)
    const float v = mine[t];
    if (p.a_cls != nullptr) p.a_cls[static_cast<size_t>(b) * M + t0 + t] = v;
    if (rank != 0) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(peer_addr(&a[t0 + t], 0)), "f"(v) : "memory");
  }
  cluster_barrier();
  if (rank != 0) return;   // CTA 0 finishes alone; no store into another CTA's memory after this point

  // Quartiles.  Each needs two neighbouring order statistics; half of the CTA finds the ones of Q1, half
  // those of Q3.  Radix passes over the (non-negative) values from the highest bit in which two of
  // them differ, until the cut bin holds few enough values to rank them against each other.
  const float pos[2] = {0.25f * static_cast<float>(M - 1), 0.75f * static_cast<float>(M - 1)};
  const int half = threadIdx.x / kHalf, th = threadIdx.x % kHalf;
  const int want = static_cast<int>(floorf(half ? pos[1] : pos[0]));
  uint32_t all_and = 0xffffffffu, all_or = 0u;
  for (int j = threadIdx.x; j < M; j += kThreads) {
    const uint32_t u = __float_as_uint(a[j]);
    all_and &= u;
    all_or |= u;
  }
  all_and = __reduce_and_sync(0xffffffffu, all_and);
  all_or = __reduce_or_sync(0xffffffffu, all_or);
  if (lane == 0) {
    band[warp] = all_and;
    bor[warp] = all_or;
  }
  __syncthreads();
  all_and = __reduce_and_sync(0xffffffffu, band[lane & (kWarps - 1)]);
  all_or = __reduce_or_sync(0xffffffffu, bor[lane & (kWarps - 1)]);
  auto meet = [&]() {   // (of this half)
    __syncwarp();
    if (half == 0) asm volatile("bar.sync 1, %0;" ::"n"(kHalf) : "memory");
    else asm volatile("bar.sync 2, %0;" ::"n"(kHalf) : "memory");
  };
  const uint32_t differ = all_and ^ all_or;
  const int hb = differ ? 31 - __clz(differ) : 7;
  uint32_t mask = hb >= 31 ? 0u : ~((2u << hb) - 1u), prefix = all_and & mask;
  int rest = want, here = 0;
  for (int shift = hb >= 7 ? hb - 7 : 0;; shift = shift > 8 ? shift - 8 : 0) {
    for (int j = th; j < M; j += kHalf) {
      const uint32_t u = __float_as_uint(a[j]);
      if ((u & mask) == prefix) atomicAdd(&hist[half][(u >> shift) & 255u], 1);
    }
    meet();
    // every warp scans the bins for itself: eight per lane
    const int4 lo = *reinterpret_cast<const int4*>(&hist[half][8 * lane]), hi = *reinterpret_cast<const int4*>(&hist[half][8 * lane + 4]);
    const int bins[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    int sum = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) sum += bins[e];
    int inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += t;
    }
    int below = inc - sum, digit = -1, off = 0, cnt = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (below <= rest && rest < below + bins[e]) {
        digit = 8 * lane + e;
        off = rest - below;
        cnt = bins[e];
      }
      below += bins[e];
    }
    const int owner = __ffs(__ballot_sync(0xffffffffu, digit >= 0)) - 1;
    digit = __shfl_sync(0xffffffffu, digit, owner);
    rest = __shfl_sync(0xffffffffu, off, owner);
    here = __shfl_sync(0xffffffffu, cnt, owner);
    prefix = (prefix & ~(255u << shift)) | (static_cast<uint32_t>(digit) << shift);
    mask |= 255u << shift;
    if (here <= kRanked || shift == 0) break;
    meet();
    hist[half][th] = 0;
    hist[half][th + kHalf] = 0;
    meet();
  }
  // the cut bin's values (beyond kRanked of them all digits are resolved and they are all the prefix),
  // and the smallest value above it
  uint32_t next = 0xffffffffu;
  for (int j = th; j < M; j += kHalf) {
    const uint32_t u = __float_as_uint(a[j]);
    if ((u & mask) > prefix) next = min(next, u);
    else if ((u & mask) == prefix && here <= kRanked) ranked[half][atomicAdd(&n_ranked[half], 1)] = u;
  }
  next = __reduce_min_sync(0xffffffffu, next);
  if (lane == 0) atomicMin(&over[half], next);
  meet();
  if (here > kRanked) {
    if (th == 0) {
      order[half][0] = prefix;
      order[half][1] = rest + 1 < here ? prefix : over[half];
    }
  } else if (th < here) {
    const uint32_t me = ranked[half][th];
    int rk = 0;
#pragma unroll 4
    for (int y = 0; y < here; ++y) {
      const uint32_t o = ranked[half][y];
      rk += o < me || (o == me && y < th) ? 1 : 0;
    }
    if (rk == rest) order[half][0] = me;
    if (rk == rest + 1) order[half][1] = me;
    if (rk == rest && rest + 1 >= here) order[half][1] = over[half];
  }
  __syncthreads();
  float quart[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const float lo = __uint_as_float(order[x][0]);
    const float hi = static_cast<int>(floorf(pos[x])) + 1 < M ? __uint_as_float(order[x][1]) : lo;
    quart[x] = lo + (hi - lo) * (pos[x] - floorf(pos[x]));
  }
  const float q1 = quart[0], q3 = quart[1];
  const float mu = q3 + 1.5f * (q3 - q1);
  if (threadIdx.x == 0 && p.mu_out != nullptr) p.mu_out[b] = mu;

  // O = { j : a[j] > mu }, ascending; at most key_max of them are stored (the lowest indices)
  const int n_word = (M + 31) / 32;
  for (int w = warp; w < n_word; w += kWarps) {
    const int j = 32 * w + lane;
    const uint32_t word = __ballot_sync(0xffffffffu, j < M && a[j] > mu);
    if (lane == 0) words[w] = word;
  }
  __syncthreads();
  int before[4], total;
  bitmap_prefix(words, lane, before, &total);
  const int slot = warp & 3, mine_before = slot == 0 ? before[0] : (slot == 1 ? before[1] : (slot == 2 ? before[2] : before[3]));
  for (int w = warp; w < n_word; w += kWarps) {   // (w & 3 is the same for all words of a warp)
    const uint32_t word = words[w];
    const int pos = __shfl_sync(0xffffffffu, mine_before, w >> 2) + __popc(word & ((1u << lane) - 1u));
    if (((word >> lane) & 1u) && pos < p.key_max) p.key_idx[static_cast<size_t>(b) * p.key_max + pos] = 32 * w + lane;
  }
  if (threadIdx.x == 0) p.key_cnt[b] = total < p.key_max ? total : p.key_max;
}

inline bool aligned16(const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; }

template <typename Kernel, typename Params>
cudaError_t launch_cluster(Kernel kernel, int batch, int cluster, size_t smem, cudaStream_t stream, const Params& p) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(batch * cluster));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

// What the calls ask a device once.  Plain words, to which every thread would store the same: the C entries take no
// lock and allocate nothing (a container's insertion may throw).
constexpr int kMaxDevices = 64;
struct DeviceFacts {
  std::atomic<int> sms;
  std::atomic<int> merge_clusters[2][kMaxMergeCluster + 1];   // clusters of the merge held at once, by FLY and size (0: not asked yet)
};
inline DeviceFacts& facts_of(int dev) {
  static DeviceFacts known[kMaxDevices + 1];               // (the last one: devices beyond, asked on every call)
  return known[dev >= 0 && dev < kMaxDevices ? dev : kMaxDevices];
}

inline int sm_count(int dev) {
  std::atomic<int>& known = facts_of(dev).sms;
  int n = known.load(std::memory_order_relaxed);
  if (n > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
    (void)cudaGetLastError();
    return 1;
  }
  if (dev >= 0 && dev < kMaxDevices) known.store(n, std::memory_order_relaxed);
  return n;
}

using MergeKernel = void (*)(MergeParams);
using KeySetKernel = void (*)(KeySetParams);

inline int resident_merge_clusters(int dev, MergeKernel kernel, int fly, int cluster) {
  std::atomic<int>& known = facts_of(dev).merge_clusters[fly - 1][cluster];
  int n = known.load(std::memory_order_relaxed);
  if (n > 0) return n;
  n = ask_resident_clusters(reinterpret_cast<const void*>(kernel), cluster, kThreads, 0);
  if (n < 1) return 1;                                     // no answer (the launch will tell): as if one fitted
  if (dev >= 0 && dev < kMaxDevices) known.store(n, std::memory_order_relaxed);
  return n;
}

inline mustdrop_status_t finish(cudaError_t e) {
  if (e == cudaSuccess) return MUSTDROP_OK;
  set_last_cuda_error(e);
  return MUSTDROP_ERR_CUDA;
}

}  // namespace
}  // namespace mustdrop

extern "C" mustdrop_status_t mustdrop_spatial_merge(int32_t batch, int32_t grid, int32_t window, int32_t channels,
                                                    float tau, const void* tokens, void* merged, int32_t* slots,
                                                    int32_t* merged_cnt, float* window_sim, void* cuda_stream) {
  using namespace mustdrop;
  if (batch <= 0 || grid <= 0 || channels <= 0 || tokens == nullptr || merged == nullptr || slots == nullptr ||
      merged_cnt == nullptr || !(tau == tau))
    return MUSTDROP_ERR_INVALID_ARG;
  if (window != 2 || (grid % 2) != 0 || grid * grid > kMaxSlots || (channels % 8) != 0 || batch > 65535)
    return MUSTDROP_ERR_UNSUPPORTED;
  const void* ptrs[] = {tokens, merged, slots, merged_cnt, window_sim};
  for (const void* q : ptrs)
    if (q != nullptr && !aligned16(q)) return MUSTDROP_ERR_INVALID_ARG;
  MergeParams p;
  p.tokens = static_cast<const uint4*>(tokens);
  p.merged = static_cast<uint4*>(merged);
  p.slots = slots; p.merged_cnt = merged_cnt; p.window_sim = window_sim;
  p.grid = grid; p.vecs = channels / 8; p.tau = tau;
  p.inv_grid = ((1u << 20) + grid - 1) / grid;
  p.inv_half = ((1u << 20) + grid / 2 - 1) / (grid / 2);
  const int n_win = (grid / 2) * (grid / 2);
  int dev = -1, resident[kMaxMergeCluster + 1] = {};
  if (cudaGetDevice(&dev) != cudaSuccess) (void)cudaGetLastError();
  const int fly = merge_fly(p.vecs);
  const MergeKernel kernel = fly == 2 ? spatial_merge_kernel<2> : spatial_merge_kernel<1>;
  for (int c = 1; c <= kMaxMergeCluster; ++c) resident[c] = resident_merge_clusters(dev, kernel, fly, c);
  const int cluster = merge_cluster(batch, n_win, resident);
  return finish(launch_cluster(kernel, batch, cluster, 0, static_cast<cudaStream_t>(cuda_stream), p));
}

extern "C" mustdrop_status_t mustdrop_key_set(int32_t batch, int32_t n_heads, int32_t head_dim, int32_t n_tokens,
                                              int32_t key_max, const void* q_cls, const void* k, float* a_cls,
                                              float* mu_out, int32_t* key_idx, int32_t* key_cnt, void* cuda_stream) {
  using namespace mustdrop;
  if (batch <= 0 || n_heads <= 0 || head_dim <= 0 || n_tokens <= 0 || key_max <= 0 || q_cls == nullptr ||
      k == nullptr || key_idx == nullptr || key_cnt == nullptr)
    return MUSTDROP_ERR_INVALID_ARG;
  if ((head_dim % 8) != 0 || head_dim > 256 || n_tokens > kMaxSlots || batch > 65535) return MUSTDROP_ERR_UNSUPPORTED;
  const void* ptrs[] = {q_cls, k, a_cls, mu_out, key_idx, key_cnt};
  for (const void* q : ptrs)
    if (q != nullptr && !aligned16(q)) return MUSTDROP_ERR_INVALID_ARG;
  KeySetParams p;
  p.q_cls = static_cast<const __nv_bfloat16*>(q_cls);
  p.k = static_cast<const uint4*>(k);
  p.a_cls = a_cls; p.mu_out = mu_out; p.key_idx = key_idx; p.key_cnt = key_cnt;
  p.H = n_heads; p.D = head_dim; p.M = n_tokens; p.key_max = key_max;
  p.scale_log2e = 1.4426950408889634f / sqrtf(static_cast<float>(head_dim));
  int cluster = 8;
  while (cluster > 1 && n_tokens < 8 * cluster) cluster >>= 1;   // 1, 2, 4 or 8 CTAs
  p.part = ((n_tokens + cluster - 1) / cluster + kParts - 1) / kParts;
  // as many heads at a time as leave four CTAs on an SM (32 KB besides the static part), at least one
  const size_t per_head = kParts * (sizeof(float2) * cluster + sizeof(float) * p.part) + sizeof(float2);
  p.block = static_cast<int>(32 * 1024 / per_head);
  if (p.block > n_heads) p.block = n_heads;
  if (p.block < 1) p.block = 1;
  const size_t smem = p.block * per_head;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) (void)cudaGetLastError();
  KeySetKernel kernel = nullptr;
  switch (key_rows(head_dim, p.part, batch * cluster, sm_count(dev))) {
    case KeyRows::kLanePerVector5: kernel = key_set_kernel<0, 1, 5, false>; break;
    case KeyRows::kLanePerVector3Ahead: kernel = key_set_kernel<0, 1, 3, true>; break;
    case KeyRows::kFour1x3Ahead: kernel = key_set_kernel<4, 1, 3, true>; break;
    case KeyRows::kFour1x5: kernel = key_set_kernel<4, 1, 5, false>; break;
    case KeyRows::kFour2x2: kernel = key_set_kernel<4, 2, 2, false>; break;
    case KeyRows::kFour2x2Ahead: kernel = key_set_kernel<4, 2, 2, true>; break;
    case KeyRows::kFour3x1Ahead: kernel = key_set_kernel<4, 3, 1, true>; break;
    case KeyRows::kEight2x2: kernel = key_set_kernel<8, 2, 2, false>; break;
    case KeyRows::kEight4x1Ahead: kernel = key_set_kernel<8, 4, 1, true>; break;
  }
  cudaError_t e = ensure_kernel_attributes(reinterpret_cast<const void*>(kernel), false);
  if (e != cudaSuccess) return finish(e);
  return finish(launch_cluster(kernel, batch, cluster, smem, static_cast<cudaStream_t>(cuda_stream), p));
}
