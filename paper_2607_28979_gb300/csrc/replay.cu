// Replay attention of the post-translation phase (App. C.4) on sm_103a: the
// Top-S selection of the source-guided layers, and V^T for the full layers.
//
//   replay_select_kernel  one warp per context row (b, u): the S positions j <= u
//                         with the largest guidance score A[b][u][j] (ties to the
//                         lower position), written in ascending order. It is exact
//                         work on the 16-bit images of the scores: a bound that at
//                         least S of the row's scores reach, taken from the maxima of
//                         groups of scores, leaves about 1.4 S candidates, and a
//                         bisection over those gives the threshold V and how many of
//                         the positions scoring V are taken. Rows with u + 1 <= S take
//                         every position.
//   replay_select_hist_kernel, for S past 416: the threshold from two histograms over
//                         the row's keys in shared memory.
//   replay_select_stream_kernel, for rows past 4,096 positions: histograms of the high
//                         and the low byte, reading the row once per pass.
//   replay_vt_kernel      V -> V^T per layer for the full-attention kernel.
//   The attention kernels are in replay_fmha.cu (full causal attention on tcgen05) and
//   replay_gather.cu (guided layers, and the full layers that tiling does not take).
#include <limits.h>
#include <string.h>

#include <algorithm>

#include "replay_common.cuh"

namespace mot {
namespace {

constexpr int kSelWarps = 8;         // rows per CTA, one warp each
constexpr int kSelCopies = 4;        // histogram copies per warp

// Warp-wide exclusive prefix of v (and the warp total).
__device__ __forceinline__ int warp_excl_scan(int v, int& total) {
  const int lane = threadIdx.x & 31;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  total = __shfl_sync(0xffffffffu, x, 31);
  return x - v;
}

// The bin of a warp's histogram (C copies of 256 bins) that holds the
// k-th largest counted key, scanning from bin 255 down: lane 0 sums the top 8
// bins, lane 31 the bottom 8. On return k is the rank left inside that bin.
template <int C = kSelCopies>
__device__ __forceinline__ uint32_t kth_bin(const int (*h)[256], int& k) {
  const int lane = threadIdx.x & 31;
  int c[8], t = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    c[e] = 0;
#pragma unroll
    for (int cp = 0; cp < C; ++cp) c[e] += h[cp][(31 - lane) * 8 + (7 - e)];
    t += c[e];
  }
  int tot;
  const int before = warp_excl_scan(t, tot);
  int found = -1, krem = 0, acc = before;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    if (found < 0 && acc + c[e] >= k) {
      found = (31 - lane) * 8 + (7 - e);
      krem = k - acc;
    }
    acc += c[e];
  }
  const int src = __ffs(__ballot_sync(0xffffffffu, found >= 0)) - 1;
  k = __shfl_sync(0xffffffffu, krem, src);
  return uint32_t(__shfl_sync(0xffffffffu, found, src));
}

// Order-preserving keys of two bf16 scores packed in a word (low half first):
// a negative score's bits are inverted, a positive score's sign bit is set.
__device__ __forceinline__ uint32_t ord16x2(uint32_t q) {
  uint32_t sign;   // 0xFFFF in each half whose sign bit is set (prmt's sign-replicating selectors)
  asm("prmt.b32 %0, %1, 0, 0xBB99;" : "=r"(sign) : "r"(q));
  return q ^ (sign | 0x80008000u);
}

// A workspace row's entries past its positions repeat them in turn: were they all one position (the
// first, which many rows hold), the gathers of a set of 100 in 128 slots would queue at its L2 slice
// (4 x 4096 positions, 12 heads of 128 on 2, S = 70: 307 us, 142 so; also rows below S, where all the
// padding was position 0: 100 positions, 28 heads on 4, S = 128: 21 us, 11 so).
__device__ __forceinline__ void pad_row(const ReplayArgs& a, int32_t* out) {   // S positions found
  const int lane = threadIdx.x & 31, S = a.d.S;
  if (a.sel_stride > S) {
    __syncwarp();
    for (int j = S + lane; j < a.sel_stride; j += 32)
      out[j] = static_cast<volatile int32_t*>(out)[(j - S) % S];
  }
}
__device__ __forceinline__ void take_all(const ReplayArgs& a, int32_t* out, int n) {   // n <= S positions
  for (int j = threadIdx.x & 31; j < a.sel_stride; j += 32) out[j] = j < n ? j : a.pad ? j % n : -1;
}

// Selection for any max_seq. One warp per context row (b, u). With o = the
// order-preserving 16 bits of a score, the S-th largest (o, -j) key is found in
// two histogram passes over o (high byte, then low byte): V = its score bits, k =
// how many positions with o == V it takes. The selection is then every o > V plus
// the k lowest positions with o == V, compacted in ascending order by warp scans.
// Each lane reads 8 consecutive scores per step (16-byte loads when max_seq % 8
// == 0); every pass reads the row again.
__global__ void __launch_bounds__(32 * kSelWarps) replay_select_stream_kernel(const ReplayArgs a) {
  pdl_enter();
  __shared__ int hist[kSelWarps][kSelCopies][256];   // copy lane % kSelCopies: fewer same-bin collisions
  const ReplayDims& d = a.d;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * kSelWarps + w;
  if (row >= d.B * d.N) return;
  const int b = row / d.N, u = row - b * d.N;
  if (u >= seq_len_of(a, b)) return;
  int32_t* out = a.sel + int64_t(row) * a.sel_stride;
  const int n = u + 1;
  if (n <= d.S) {
    take_all(a, out, n);
    return;
  }
  const uint16_t* A = static_cast<const uint16_t*>(a.guide) + int64_t(row) * d.N;
  const bool vec = (d.N & 7) == 0;   // then every 8-score group of the row is 16-byte aligned
  // the 8 order-preserving scores at positions j8 .. j8 + 7 (0 past n; never counted)
  auto load8 = [&](int j8, uint32_t (&o)[8]) {
    if (vec) {
      const uint4 q = __ldg(reinterpret_cast<const uint4*>(A + j8));
      const uint32_t qq[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        o[2 * e] = ord16(qq[e] & 0xFFFFu);
        o[2 * e + 1] = ord16(qq[e] >> 16);
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = j8 + e < n ? ord16(__ldg(A + j8 + e)) : 0u;
    }
  };
  int* hw = hist[w][lane % kSelCopies];
  int k = d.S;
  uint32_t hi = 0, V = 0;
  for (int pass = 0; pass < 2; ++pass) {
    for (int i = lane; i < kSelCopies * 256; i += 32) hist[w][0][i] = 0;
    __syncwarp();
    for (int j8 = lane * 8; j8 - lane * 8 < n; j8 += 256) {   // warp-uniform trip count
      uint32_t o[8];
      if (j8 < n) load8(j8, o);
      if (pass == 0) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (j8 + e < n) atomicAdd(&hw[o[e] >> 8], 1);
      } else {
        // only the scores in bin `hi` count, spread over 256 low bytes
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (j8 + e < n && (o[e] >> 8) == hi) atomicAdd(&hw[o[e] & 0xFFu], 1);
      }
    }
    __syncwarp();
    const uint32_t bin = kth_bin(hist[w], k);
    if (pass == 0)
      hi = bin;
    else
      V = (hi << 8) | bin;   // k: positions with o == V to take, lowest first
    __syncwarp();
  }
  // compaction in ascending position order, 256 positions per round
  int base = 0, eq_taken = 0;
  for (int j8 = lane * 8; j8 - lane * 8 < n; j8 += 256) {
    uint32_t o[8];
    if (j8 < n) load8(j8, o);
    int n_eq = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) n_eq += (j8 + e < n && o[e] == V);
    int eq_tot;
    int eq_rank = eq_taken + warp_excl_scan(n_eq, eq_tot);
    bool sel[8];
    int n_sel = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const bool in = j8 + e < n;
      const bool eq = in && o[e] == V;
      sel[e] = in && (o[e] > V || (eq && eq_rank < k));
      eq_rank += eq;
      n_sel += sel[e];
    }
    int sel_tot;
    int pos = base + warp_excl_scan(n_sel, sel_tot);
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (sel[e]) out[pos++] = j8 + e;
    base += sel_tot;
    eq_taken += eq_tot;
  }
  pad_row(a, out);
}

// Selection for max_seq <= 4096 and sets past kSelTwoSets (where too many keys pass the bound of
// replay_select_kernel), with the row's keys cached in shared memory.
// One warp per context row (b, u): the row is read once and turned into
// order-preserving keys o (lane L holds positions 256 r + 8 L + e, as one 16-byte
// word of packed keys per round r), together with its key range [omin, omax].
// The S-th largest (o, -j) key is then found by a radix selection over o - omin:
// a 256-bin histogram of the top digit (o - omin) >> sh, sh the smallest shift
// that fits the row's range into 256 bins, then, when sh > 0, a histogram of the
// low sh bits among the keys of the chosen bin. That gives V, the threshold key,
// and k, how many positions with o == V are taken. The compaction keeps every
// o > V and the k lowest positions with o == V, in ascending order. The digits
// follow the row's own range, so increments spread over many bins even when the
// scores share a few binades.
constexpr int kSelCacheWarps = 4;    // rows per CTA
constexpr int kSelCacheRounds = 16;  // 256-position rounds cached per row: max_seq <= 4096
constexpr int kSelCacheCopies = 1;   // histogram copies per warp (36 KB per CTA: 6 CTAs per SM)

__global__ void __launch_bounds__(32 * kSelCacheWarps) replay_select_hist_kernel(const ReplayArgs a) {
  pdl_enter();
  __shared__ int hist[kSelCacheWarps][kSelCacheCopies][256];   // copy lane % kSelCacheCopies
  __shared__ uint4 keys[kSelCacheWarps][kSelCacheRounds][32];
  const ReplayDims& d = a.d;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = blockIdx.x * kSelCacheWarps + w;
  if (row >= d.B * d.N) return;
  const int b = row / d.N, u = row - b * d.N;
  if (u >= seq_len_of(a, b)) return;
  int32_t* out = a.sel + int64_t(row) * a.sel_stride;
  const int n = u + 1;
  if (n <= d.S) {
    take_all(a, out, n);
    return;
  }
  const uint16_t* A = static_cast<const uint16_t*>(a.guide) + int64_t(row) * d.N;
  const bool vec = (d.N & 7) == 0;   // then every 8-score group of the row is 16-byte aligned
  const int nr = (n + 255) >> 8;     // rounds holding positions < n (<= kSelCacheRounds)
  uint4 (*kc)[32] = keys[w];
  uint32_t lo = 0xFFFFu, hi = 0u;
  // Rounds r < nfull hold n's positions on every lane (no per-position test there).
  const int nfull = n >> 8;
  int r0 = 0;
  if (vec) {
    uint32_t lo1 = 0xFFFFu, hi1 = 0u;
#pragma unroll 4
    for (; r0 < nfull; ++r0) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(A + r0 * 256 + lane * 8));
      const uint32_t q[4] = {ord16x2(v.x), ord16x2(v.y), ord16x2(v.z), ord16x2(v.w)};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        lo = min(lo, q[i] & 0xFFFFu);
        hi = max(hi, q[i] & 0xFFFFu);
        lo1 = min(lo1, q[i] >> 16);
        hi1 = max(hi1, q[i] >> 16);
      }
      kc[r0][lane] = make_uint4(q[0], q[1], q[2], q[3]);
    }
    lo = min(lo, lo1);
    hi = max(hi, hi1);
  }
#pragma unroll 4
  for (int r = r0; r < nr; ++r) {
    const int j8 = r * 256 + lane * 8;
    const int lim = min(n - j8, 8);   // this lane's positions < n in the round (may be <= 0)
    uint32_t q[4] = {0u, 0u, 0u, 0u};
    if (lim > 0) {
      if (vec) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(A + j8));
        q[0] = v.x;
        q[1] = v.y;
        q[2] = v.z;
        q[3] = v.w;
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (e < lim) q[e >> 1] |= uint32_t(__ldg(A + j8 + e)) << (16 * (e & 1));
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      q[i] = ord16x2(q[i]);
      const uint32_t o0 = q[i] & 0xFFFFu, o1 = q[i] >> 16;
      if (2 * i < lim) {
        lo = min(lo, o0);
        hi = max(hi, o0);
      }
      if (2 * i + 1 < lim) {
        lo = min(lo, o1);
        hi = max(hi, o1);
      }
    }
    kc[r][lane] = make_uint4(q[0], q[1], q[2], q[3]);
  }
  const uint32_t omin = __reduce_min_sync(0xffffffffu, lo);
  const uint32_t range = __reduce_max_sync(0xffffffffu, hi) - omin;   // < 65536
  const int sh = range > 255u ? 24 - __clz(range) : 0;   // (range >> sh) <= 255, sh <= 8
  int* hw = hist[w][lane % kSelCacheCopies];
  int k = d.S;
  // key e (0..7) of a lane's 16-byte word
  auto key_of = [](const uint4& v, int e) -> uint32_t {
    const uint32_t x = e < 2 ? v.x : e < 4 ? v.y : e < 6 ? v.z : v.w;
    return (e & 1) ? x >> 16 : x & 0xFFFFu;
  };
  // Every key is at least omin, so subtracting omin from both halves of a packed word
  // borrows nothing across them: each half holds its own o - omin.
  const uint32_t omin2 = omin * 0x10001u;
  // top digit
  for (int i = lane; i < kSelCacheCopies * 256; i += 32) hist[w][0][i] = 0;
  __syncwarp();
  for (int r = 0; r < nfull; ++r) {
    const uint4 v = kc[r][lane];
    const uint32_t wd[4] = {v.x - omin2, v.y - omin2, v.z - omin2, v.w - omin2};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      atomicAdd(&hw[(wd[i] & 0xFFFFu) >> sh], 1);
      atomicAdd(&hw[wd[i] >> (16 + sh)], 1);
    }
  }
  if (nfull < nr) {
    const int lim = min(n - (nfull * 256 + lane * 8), 8);
    const uint4 v = kc[nfull][lane];
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (e < lim) atomicAdd(&hw[(key_of(v, e) - omin) >> sh], 1);
  }
  __syncwarp();
  const uint32_t top = kth_bin<kSelCacheCopies>(hist[w], k);
  uint32_t V = omin + (top << sh);
  if (sh > 0) {   // the low sh bits among the keys of bin `top`: o - omin in [top << sh, + 2^sh)
    __syncwarp();
    for (int i = lane; i < kSelCacheCopies * 256; i += 32) hist[w][0][i] = 0;
    __syncwarp();
    const uint32_t msk = (1u << sh) - 1u, lo_b = top << sh;
    for (int r = 0; r < nfull; ++r) {
      const uint4 v = kc[r][lane];
      const uint32_t wd[4] = {v.x - omin2, v.y - omin2, v.z - omin2, v.w - omin2};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t a = wd[i] & 0xFFFFu, c = wd[i] >> 16;
        if (a - lo_b <= msk) atomicAdd(&hw[a & msk], 1);
        if (c - lo_b <= msk) atomicAdd(&hw[c & msk], 1);
      }
    }
    if (nfull < nr) {
      const int lim = min(n - (nfull * 256 + lane * 8), 8);
      const uint4 v = kc[nfull][lane];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const uint32_t o = key_of(v, e) - omin;
        if (e < lim && (o >> sh) == top) atomicAdd(&hw[o & msk], 1);
      }
    }
    __syncwarp();
    V += kth_bin<kSelCacheCopies>(hist[w], k);
  }
  // compaction in ascending position order; bit e of a lane's masks is position 256 r + 8 lane + e
  int base = 0, eq_taken = 0;
  for (int r = 0; r < nr && base < d.S; ++r) {   // warp-uniform
    const int j8 = r * 256 + lane * 8;
    const uint4 v = kc[r][lane];
    uint32_t gt = 0u, eq = 0u;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint32_t o = key_of(v, e);
      gt |= uint32_t(o > V) << e;
      eq |= uint32_t(o == V) << e;
    }
    if (r == nfull) {   // the partial round: positions past n never count
      const int lim = min(n - j8, 8);
      const uint32_t in = lim <= 0 ? 0u : (1u << lim) - 1u;
      gt &= in;
      eq &= in;
    }
    uint32_t sel = gt;
    if (__any_sync(0xffffffffu, eq != 0u)) {   // the k lowest positions at the threshold are taken
      int eq_tot;
      int take = k - (eq_taken + warp_excl_scan(__popc(eq), eq_tot));
      for (uint32_t m = eq; m != 0u && take > 0; m &= m - 1u, --take) sel |= m & (0u - m);
      eq_taken += eq_tot;
    }
    int sel_tot;
    int pos = base + warp_excl_scan(__popc(sel), sel_tot);
    for (uint32_t m = sel; m != 0u; m &= m - 1u) out[pos++] = j8 + __ffs(m) - 1;
    base += sel_tot;
  }
  pad_row(a, out);
}

// ---------------------------------------------------------------- rows of up to 4,096 positions
//
// A row is read in 16-byte words, 256 positions per round: lane L's word of round r holds
// positions 256 r + 8 L + e - off, e = 0..7, where off is how far the row starts past a
// 16-byte boundary, so that rows of any max_seq are read in whole words. Slots of a word
// outside the row hold key 0.
struct RowWords {
  const uint16_t* A;   // the 16-byte boundary at or before the row
  int off, end;        // the row is slots off .. end - 1 of its words
  int r0, nfull, nr;   // of nr rounds, r0 .. nfull - 1 are inside the row on every lane

  __device__ __forceinline__ RowWords(const ReplayArgs& a, int row, int n) {
    const int64_t at = int64_t(row) * a.d.N;   // the guide itself is 16-byte aligned
    off = static_cast<int>(at & 7);
    A = static_cast<const uint16_t*>(a.guide) + (at - off);
    end = n + off;
    r0 = off == 0 ? 0 : 1;
    nfull = end >> 8;
    nr = (end + 255) >> 8;
  }
  __device__ __forceinline__ const uint16_t* word(int r) const {
    return A + r * 256 + (threadIdx.x & 31) * 8;
  }
  __device__ __forceinline__ uint32_t in(int r) const {   // valid slots of this lane's word
    const int j8 = r * 256 + (threadIdx.x & 31) * 8, lim = end - j8;
    uint32_t m = lim >= 8 ? 0xFFu : lim <= 0 ? 0u : (1u << lim) - 1u;
    if (j8 == 0) m &= 0xFFu << off;
    return m;
  }
  // RAW: the scores' own bits instead of the order-preserving keys (rows without sign bits)
  template <bool RAW>
  __device__ __forceinline__ void whole(int r, uint32_t (&q)[4]) const {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(word(r)));
    q[0] = RAW ? v.x : ord16x2(v.x);
    q[1] = RAW ? v.y : ord16x2(v.y);
    q[2] = RAW ? v.z : ord16x2(v.z);
    q[3] = RAW ? v.w : ord16x2(v.w);
  }
  // a round with slots outside the row on some lanes; m: the valid slots
  template <bool RAW>
  __device__ __forceinline__ void edge(int r, uint32_t (&q)[4], uint32_t& m) const {
    m = in(r);
    if (m == 0xFFu) {
      whole<RAW>(r, q);
      return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = 0u;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (m >> e & 1u) {
        const uint16_t x = __ldg(word(r) + e);
        q[e >> 1] |= (RAW ? uint32_t(x) : ord16(x)) << (16 * (e & 1));
      }
  }
};

constexpr int kSelRowWarps = 4;
constexpr int kSelRowCtas = 10;      // CTAs per SM (up to 51 registers a thread)
constexpr int kSelRowSeq = 4096;     // largest max_seq taken
constexpr int kSelOneSet = 160;      // largest S taken with 256 group maxima
constexpr int kSelTwoSets = 416;     // largest S taken with 512: four rows of 4,096, S = 416: 66 us (75 by
                                     // histograms), 432: 79 (75), 448: 97 (74); of 1,024: equal

// Keys of packed pairs against a threshold key. RAW keys are non-negative bf16 bits below the
// NaNs, which order as the numbers they are: one packed comparison per pair.
__device__ __forceinline__ uint32_t ge_pair(uint32_t q, uint32_t key2) {   // 0xFFFF per half
  __nv_bfloat162 x, y;
  memcpy(&x, &q, 4);
  memcpy(&y, &key2, 4);
  return __hge2_mask(x, y);
}

// 8 x the number of keys >= key among NW packed pairs.
template <bool RAW, int NW>
__device__ __forceinline__ int count_ge8(const uint32_t* q, uint32_t key) {
  int c = 0;
  if (RAW) {
    const uint32_t key2 = key * 0x10001u;
#pragma unroll
    for (int i = 0; i < NW; i += 2)
      c += __popc(__byte_perm(ge_pair(q[i], key2), ge_pair(q[i + 1], key2), 0x6420));
  } else {
    const uint32_t t = key << 16;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      c += (q[i] << 16) >= t;
      c += q[i] >= t;
    }
    c *= 8;
  }
  return c;
}

// Bits e of a word's keys >= key.
template <bool RAW>
__device__ __forceinline__ uint32_t ge_bits(const uint32_t (&q)[4], uint32_t key) {
  if (RAW) {
    const uint32_t key2 = key * 0x10001u;
    const uint32_t x = __byte_perm(ge_pair(q[0], key2), ge_pair(q[1], key2), 0x6420);
    const uint32_t y = __byte_perm(ge_pair(q[2], key2), ge_pair(q[3], key2), 0x6420);
    return (((x & 0x08040201u) | (y & 0x80402010u)) * 0x01010101u) >> 24;
  }
  const uint32_t t = key << 16;
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if ((q[i] << 16) >= t) m |= 1u << (2 * i);
    if (q[i] >= t) m |= 2u << (2 * i);
  }
  return m;
}

// Every key above V and the lowest k positions at V, in ascending order: S positions.
template <bool RAW>
__device__ __noinline__ void select_at(const RowWords w, uint32_t V, int k, int S, int32_t* out) {
  const int lane = threadIdx.x & 31;
  int base = 0, eq_taken = 0;
  for (int r = 0; r < w.nr && base < S; ++r) {   // warp-uniform
    uint32_t q[4], in = 0xFFu;
    if (r >= w.r0 && r < w.nfull) w.whole<RAW>(r, q);
    else w.edge<RAW>(r, q, in);
    uint32_t sel = V == 0xFFFFu ? 0u : ge_bits<RAW>(q, V + 1u) & in;
    const uint32_t eq = ge_bits<RAW>(q, V) & in & ~sel;
    if (__any_sync(0xffffffffu, eq != 0u)) {   // the k lowest positions at the threshold are taken
      int eq_tot;
      int take = k - (eq_taken + warp_excl_scan(__popc(eq), eq_tot));
      for (uint32_t m = eq; m != 0u && take > 0; m &= m - 1u, --take) sel |= m & (0u - m);
      eq_taken += eq_tot;
    }
    int sel_tot;
    int pos = base + warp_excl_scan(__popc(sel), sel_tot);
    for (uint32_t m = sel; m != 0u; m &= m - 1u)
      out[pos++] = r * 256 + lane * 8 + __ffs(m) - 1 - w.off;
    base += sel_tot;
  }
}

// The selection by bisection over all of the row's keys, which sit in L1: at least S of them
// reach lo >= 1, none reaches hi.
template <bool RAW>
__device__ __noinline__ void select_by_bisection(const RowWords w, uint32_t lo, uint32_t hi, int S,
                                                 int32_t* out) {
  int c_hi = 0, c_lo = INT_MAX;
  while (hi - lo > 1u && c_lo != S) {
    const uint32_t mid = (lo + hi) >> 1;   // >= 1: the key 0 of slots outside the row never counts
    int c = 0;
#pragma unroll 4
    for (int r = w.r0; r < w.nfull; ++r) {
      uint32_t q[4];
      w.whole<RAW>(r, q);
      c += count_ge8<RAW, 4>(q, mid);
    }
    for (int r = 0; r < w.nr; ++r) {
      if (r >= w.r0 && r < w.nfull) continue;
      uint32_t q[4], m;
      w.edge<RAW>(r, q, m);
      c += count_ge8<RAW, 4>(q, mid);
    }
    c = __reduce_add_sync(0xffffffffu, c) >> 3;
    if (c >= S) {
      lo = mid;
      c_lo = c;
    } else {
      hi = mid;
      c_hi = c;
    }
  }
  select_at<RAW>(w, lo, c_lo == S ? INT_MAX : S - c_hi, S, out);
}

// The bounded selection of one row (its steps are at replay_select_kernel). False, for RAW,
// when the row holds a sign bit or a NaN.
template <int SETS, bool RAW>
__device__ __forceinline__ bool select_bounded(const RowWords& rw, uint16_t* list, int S,
                                                       int32_t* out) {
  constexpr int CAP = 512 * SETS;
  const int lane = threadIdx.x & 31;
  // ---- 1. group maxima
  uint32_t mx[4 * SETS], sgn = 0u;
#pragma unroll
  for (int i = 0; i < 4 * SETS; ++i) mx[i] = 0u;
  auto take = [&](int set, const uint32_t (&q)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) mx[4 * set + i] = __vmaxu2(mx[4 * set + i], q[i]);
    if (RAW) sgn |= q[0] | q[1] | q[2] | q[3];
  };
  uint32_t q[4], in;
  if (rw.r0 == 1) {
    rw.edge<RAW>(0, q, in);
    take(0, q);
  }
  int r = rw.r0;
  for (; r + 4 <= rw.nfull; r += 4) {
    uint32_t x[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) rw.whole<RAW>(r + i, x[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) take(i % SETS, x[i]);
  }
  for (; r < rw.nfull; ++r) {
    rw.whole<RAW>(r, q);
    if (SETS == 1 || !(r & 1)) take(0, q);
    else take(SETS - 1, q);
  }
  for (; r < rw.nr; ++r) {
    rw.edge<RAW>(r, q, in);
    take(0, q);
  }
  // ---- 2. a key that S group maxima reach
  uint32_t lo2 = mx[0], hi2 = mx[0];
#pragma unroll
  for (int i = 1; i < 4 * SETS; ++i) {
    lo2 = __vminu2(lo2, mx[i]);
    hi2 = __vmaxu2(hi2, mx[i]);
  }
  uint32_t lo = __reduce_min_sync(0xffffffffu, min(lo2 & 0xFFFFu, lo2 >> 16));
  uint32_t hi = __reduce_max_sync(0xffffffffu, max(hi2 & 0xFFFFu, hi2 >> 16));
  if (RAW && (hi > 0x7F80u || __any_sync(0xffffffffu, (sgn & 0x80008000u) != 0u)))
    return false;
  const uint32_t kmax = ++hi;   // at least S maxima reach lo, none reaches hi
  while (hi - lo > 1u) {
    const uint32_t mid = (lo + hi) >> 1;
    const int c = __reduce_add_sync(0xffffffffu, count_ge8<RAW, 4 * SETS>(mx, mid));
    if (c >= 8 * S) {
      lo = mid;
      if (c <= 8 * (S + 16)) break;
    } else {
      hi = mid;
    }
  }
  const uint32_t L = max(lo, 1u);   // key 0 also fills the slots outside the row
  // ---- 3. candidates, two rounds per prefix sum
  int C = 0;
  auto mask = [&](int rr) -> uint32_t {
    if (rr >= rw.r0 && rr < rw.nfull) rw.whole<RAW>(rr, q);   // warp-uniform
    else rw.edge<RAW>(rr, q, in);
    return ge_bits<RAW>(q, L);
  };
  for (r = 0; r < rw.nr; r += 2) {
    const uint32_t m0 = mask(r), m1 = r + 1 < rw.nr ? mask(r + 1) : 0u;
    // inclusive prefix sums of both rounds' counts over the lanes: a lane fills its part of
    // the list from the end, highest slot first
    const int n01 = __popc(m0) | __popc(m1) << 16;
    int tot;
    const int inc = warp_excl_scan(n01, tot) + n01;
    const int c0 = tot & 0xFFFF, c1 = tot >> 16;
    if (C + c0 + c1 > CAP) {   // warp-uniform: many keys at the bound
      select_by_bisection<RAW>(rw, L, kmax, S, out);
      return true;
    }
    const int j8 = r * 256 + lane * 8;
    uint16_t* p = list + C + (inc & 0xFFFF);
    for (uint32_t m = m0; m != 0u;) {
      const int e = 31 - __clz(m);
      *--p = static_cast<uint16_t>(j8 + e);
      m ^= 1u << e;
    }
    p = list + C + c0 + (inc >> 16);
    for (uint32_t m = m1; m != 0u;) {
      const int e = 31 - __clz(m);
      *--p = static_cast<uint16_t>(j8 + 256 + e);
      m ^= 1u << e;
    }
    C += c0 + c1;
  }
  __syncwarp();
  if (C < S) {   // the bound was key 0: every other key is selected, the rest are keys of 0
    select_at<RAW>(rw, 0u, S - C, S, out);
    return true;
  }
  // ---- 4. the S-th largest candidate key V, and how many positions at V are taken
  constexpr int RK = CAP / 32;   // candidates per lane, two to a register
  const int ni = (C + 31) >> 5;  // 32-candidate groups
  uint32_t ck[RK / 2];
#pragma unroll
  for (int i = 0; i < RK / 2; ++i) {
    ck[i] = 0u;
    if (2 * i < ni) {   // warp-uniform
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int at = (2 * i + h) * 32 + lane;
        if (at < C) {
          const uint16_t x = __ldg(rw.A + list[at]);
          ck[i] |= (RAW ? uint32_t(x) : ord16(x)) << (16 * h);
        }
      }
    }
  }
  lo = L;       // C >= S candidates reach lo
  hi = kmax;    // fewer than S reach hi
  int c_lo = C, c_hi = 0;
  while (hi - lo > 1u && c_lo != S) {
    const uint32_t mid = (lo + hi) >> 1;
    int c = count_ge8<RAW, RK / 4>(ck, mid);
    if (ni > RK / 2) c += count_ge8<RAW, RK / 4>(ck + RK / 4, mid);
    c = __reduce_add_sync(0xffffffffu, c) >> 3;
    if (c >= S) {
      lo = mid;
      c_lo = c;
    } else {
      hi = mid;
      c_hi = c;
    }
  }
  const uint32_t V = lo;
  // c_lo == S: every candidate at V or above; else c_hi of them are above V = hi - 1
  const int k = c_lo == S ? INT_MAX : S - c_hi;
  // ---- 5. output
  const uint32_t below = (1u << lane) - 1u;
  int base = 0, eq_taken = 0;
#pragma unroll
  for (int i = 0; i < RK; ++i) {
    if (i >= ni) break;
    const uint32_t key = (i & 1) ? ck[i >> 1] >> 16 : ck[i >> 1] & 0xFFFFu;   // 0 past the list
    const uint32_t eq = __ballot_sync(0xffffffffu, key == V);
    const bool s = key > V || (key == V && eq_taken + __popc(eq & below) < k);
    const uint32_t m = __ballot_sync(0xffffffffu, s);
    if (s) out[base + __popc(m & below)] = list[i * 32 + lane] - rw.off;
    base += __popc(m);
    eq_taken += __popc(eq);
  }
  return true;
}

// Selection for S up to kSelTwoSets. One warp per context row (b, u); the row is read from
// global memory twice, the second time from L1.
//
//   1. Maxima: each lane keeps the maximum of every column e over the rounds: the maxima of
//      256 disjoint groups of keys (SETS = 2: 512, even and odd rounds apart).
//   2. Bound: at least S of the row's keys reach L, the S-th largest group maximum, so every
//      selected key does (a few bisection steps; any L that S to S + 16 maxima reach will do).
//   3. Candidates: the positions with keys >= L, in ascending order, about 1.4 S of them.
//   4. Threshold: bisection over the candidates' keys, held in registers, for the key V of
//      the S-th largest and the number k of positions at V taken (the lowest).
//   5. Output: the candidates above V and the first k at V, by ballots, 32 at a time.
//
// Scores without sign bits or NaNs (attention weights) are compared as bf16 pairs; other rows
// start over on their order-preserving keys. Rows with more candidates than the list holds
// (many equal scores) bisect over the whole row.
//
// Persistent: every warp walks rows, the longest first, so that the short rows fill the end.
//
// What bounds it: instruction issue and the latency of its dependent steps (1,650 warp
// instructions per row of 2,048 scores on average, 40% of the issue slots; HBM at 1.3 TB/s).
// Four rows of 4,096, one warp each, S = 128: 67.7 us with the histograms over every key
// (2,790 instructions per row), 57 us with this bound over order-preserving keys in shared
// memory, 43 us reading the row twice and comparing bf16 pairs, 40.7 us persistent. S = 32:
// 64 to 35 us; S = 256: 70 to 49 us; rows of 4,095, which the histogram kernel read one
// score at a time: 86 to 42 us; scores with sign bits: 62 to 55 us; rows of 97% zeros: 74 to
// 56 us. 512 maxima for S past 160: with 256 the bound would sit near the smallest of them.
template <int SETS>
__global__ void __launch_bounds__(32 * kSelRowWarps, kSelRowCtas)
    replay_select_kernel(const ReplayArgs a) {
  pdl_enter();
  constexpr int CAP = 512 * SETS;
  __shared__ uint16_t lists[kSelRowWarps][CAP];   // candidate slots, ascending
  const ReplayDims& d = a.d;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int step = gridDim.x * kSelRowWarps;
  for (int at = blockIdx.x * kSelRowWarps + w; at < d.B * d.N; at += step) {
    const int v = at / d.B, b = at - v * d.B, u = d.N - 1 - v;
    if (u >= seq_len_of(a, b)) continue;
    const int row = b * d.N + u;
    int32_t* out = a.sel + int64_t(row) * a.sel_stride;
    const int n = u + 1;
    if (n <= d.S) {
      take_all(a, out, n);
      continue;
    }
    const RowWords rw(a, row, n);
    __syncwarp();   // the list's last readers are done
    if (!select_bounded<SETS, true>(rw, lists[w], d.S, out))
      select_bounded<SETS, false>(rw, lists[w], d.S, out);
    pad_row(a, out);
  }
}

// ---------------------------------------------------------------- V^T for the tensor-core path

// vt[(b * Hkv + hk) * d + i][j] = v[(b * Hkv + hk) * N + j][i], 64 x 64 tiles through SMEM
// (N % 8 == 0). A thread reads 16 bytes of a row, writes its eight values as a column of the
// transposed tile in 4-byte pairs of rows, and stores 16 bytes of a transposed row: 33.6 MB for
// 4 x 4096 positions and 2 heads of 128 in 9.2 us (15.6 us with one value per thread and step).
__global__ void __launch_bounds__(256) replay_vt_kernel(const uint16_t* __restrict__ v,
                                                         uint16_t* __restrict__ vt, int N, int D) {
  pdl_enter();
  constexpr int kLd = 66;   // rows of 33 words: a column of words in 32 banks
  __shared__ __align__(4) uint16_t tile[64 * kLd];   // [i][j]
  const int bh = blockIdx.z;
  const int j0 = blockIdx.x * 64, i0 = blockIdx.y * 64;
  const uint16_t* src = v + int64_t(bh) * N * D;
  uint16_t* dst = vt + int64_t(bh) * D * N;
  {   // thread: rows j0 + 2 jp, + 1 and dims i0 + 8 c .. + 7
    const int jp = threadIdx.x & 31, c = threadIdx.x >> 5;
    const int j = j0 + 2 * jp;
    uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
    if (j < N) a = __ldg(reinterpret_cast<const uint4*>(src + int64_t(j) * D + i0 + 8 * c));
    if (j + 1 < N) b = __ldg(reinterpret_cast<const uint4*>(src + int64_t(j + 1) * D + i0 + 8 * c));
    const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {b.x, b.y, b.z, b.w};
    uint32_t* t32 = reinterpret_cast<uint32_t*>(tile);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      t32[(8 * c + 2 * k) * (kLd / 2) + jp] = __byte_perm(aw[k], bw[k], 0x5410);
      t32[(8 * c + 2 * k + 1) * (kLd / 2) + jp] = __byte_perm(aw[k], bw[k], 0x7632);
    }
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 2; ++s) {   // 512 pieces of 8 positions, eight threads per row
    const int e = s * 256 + threadIdx.x, i = e >> 3, j = (e & 7) * 8;
    const uint32_t* t32 = reinterpret_cast<const uint32_t*>(tile + i * kLd + j);
    if (j0 + j < N)
      *reinterpret_cast<uint4*>(dst + int64_t(i0 + i) * N + j0 + j) =
          make_uint4(t32[0], t32[1], t32[2], t32[3]);
  }
}
}  // namespace

bool replay_supported(const ReplayDims& d) {
  return d.Hkv > 0 && d.Hq % d.Hkv == 0 && group_ok(d.Hq / d.Hkv) &&
         (d.d == 64 || d.d == 128) && d.S >= 1 && d.S <= 4096 && d.N >= 1 && d.N <= 65536;
}

cudaError_t launch_replay_select(const ReplayArgs& a, int num_sms, cudaStream_t st) {
  const int rows = a.d.B * a.d.N;
  if (rows <= 0) return cudaSuccess;
  const int grid = std::min((rows + kSelRowWarps - 1) / kSelRowWarps, num_sms * kSelRowCtas);
  if (a.d.N > kSelRowSeq)
    replay_select_stream_kernel<<<(rows + kSelWarps - 1) / kSelWarps, 32 * kSelWarps, 0, st>>>(a);
  else if (a.d.S <= kSelOneSet)
    replay_select_kernel<1><<<grid, 32 * kSelRowWarps, 0, st>>>(a);
  else if (a.d.S <= kSelTwoSets)
    replay_select_kernel<2><<<grid, 32 * kSelRowWarps, 0, st>>>(a);
  else
    replay_select_hist_kernel<<<(rows + kSelCacheWarps - 1) / kSelCacheWarps, 32 * kSelCacheWarps,
                                0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_replay_vt(const ReplayArgs& a, void* vt, cudaStream_t st) {
  const ReplayDims& d = a.d;
  dim3 grid((d.N + 63) / 64, d.d / 64, d.B * d.Hkv);   // d is 64 or 128
  replay_vt_kernel<<<grid, 256, 0, st>>>(static_cast<const uint16_t*>(a.v),
                                         static_cast<uint16_t*>(vt), d.N, d.d);
  return cudaGetLastError();
}
}  // namespace mot
