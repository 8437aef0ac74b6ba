// SIMT translation path: plain fp32 FMA GEMMs (no TF32, no tensor cores).
// Used for fp32 caches, where the accuracy target needs true fp32 products,
// and for bf16 shapes that the tcgen05 tiling does not cover.
//
//   GEMM1:  a2[row][j] = GELU(z_row . W1cat[j] + b1[j]) * gate[row][j / H]
//   GEMM2:  y[row][c]  = a2[row] . W2cat[c] + sum_m gate[row][m] * b2[m][c]
//           stored into the target cache at (layer, b, c / d_t, s, c % d_t).
// GELU is the exact erf form; a2 is kept in fp32.
//
// One kernel for both: a CTA computes 64 rows x 32 columns with four groups of 64
// threads, each group taking a quarter of every K block; a thread accumulates 8 x 4
// outputs. Both operands sit in shared memory as their K-contiguous rows, so a 16-byte
// read holds four K values of a row and feeds two packed FMAs (fma.rn.f32x2, even and odd
// K in the halves): 64 of them per 12 reads. The groups' partial sums are added in order
// at the end. Three K blocks are in flight (cp.async for fp32 rows).
//
// What bounds it: one 64-token context (4 layers, E = 2, 768-768-768) is 2.42 GFLOP, 32 us
// at 128 FMA per SM and clock, on 384 CTAs each (the second GEMM's 192 tiles split over pairs);
// the 16-byte reads take the load path for 1.5 times the FMAs' cycles. Measured there: 160
// and 209 us as 64 x 64 tiles of 4 x 4 threads (two scalar-fed reads per 16 FMAs, half of the
// SMs idle), 49 and 59 us as 64 x 32 tiles, 49 and 50 us with the pairs; 8 x 8 outputs a thread
// took 55 and 67 us with packed pairs (one CTA per SM) and 54 and 58 us with single FMAs.
#include <cuda_bf16.h>

#include <type_traits>

#include "gelu.cuh"
#include "mot_internal.h"
#include "ptx.cuh"

namespace mot {
namespace {

constexpr int BM = 64, BN = 32, BK = 64;
constexpr int kKGroups = 4, kSimtThreads = 64 * kKGroups;
constexpr int kSimtStages = 3;
constexpr int kLd = BK + 4;   // floats per shared-memory row: 8 rows' 16-byte pieces in 8 bank groups
constexpr int kStageFloats = (BM + BN) * kLd;
constexpr int kSimtSmem = kSimtStages * kStageFloats * 4;
static_assert(BM * BN * kKGroups <= kSimtStages * kStageFloats, "partial sums reuse the stages");

__device__ __forceinline__ float ld_f(const float* p) { return __ldg(p); }
__device__ __forceinline__ float ld_f(const __nv_bfloat16* p) {
  return __bfloat162float(__ushort_as_bfloat16(__ldg(reinterpret_cast<const uint16_t*>(p))));
}
__device__ __forceinline__ float ld_a2(const float* p) { return ld_chain(p); }   // GEMM1 writes it
__device__ __forceinline__ float ld_a2(const __nv_bfloat16*) { return 0.f; }      // never: a2 is fp32
__device__ __forceinline__ void st_v(float* p, float v) { *p = v; }
__device__ __forceinline__ void st_v(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }

// Four K-consecutive values into shared memory, aligned to four in the source.
__device__ __forceinline__ void put4(float* dst, const float* src) {
  cp_async_16(smem_u32(dst), src);
}
__device__ __forceinline__ void put4(float* dst, const __nv_bfloat16* src) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(src));
  *reinterpret_cast<float4*>(dst) =
      make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u),
                  __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
}
__device__ __forceinline__ void put_zero4(float* dst) {
  *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
}

// acc (two fp32 halves) += a * b, half by half.
__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ void ld_pairs(uint32_t addr, uint64_t& a, uint64_t& b) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
}

__device__ __forceinline__ float ld_peer(uint32_t addr) {   // another CTA's shared memory
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

// GEMM 1 or 2. Grid (2 * tiles_max, columns / 32, gp * KS): blockIdx.x is a 64-row half tile.
// VEC: d_s and both K lengths are multiples of four, so every four-value piece is aligned and
// inside one row and head; otherwise values are read one by one, all of a piece's loads in flight (one
// at a time took 883 us for 2,000 tokens of 350 -> 802 -> 132 and 3 layers, E = 2; 557 now, and 635 with
// 64 x 64 tiles). KS = 2 (GEMM2): a cluster of two
// CTAs, each with half of the K blocks; each then sums and stores half of the tile's rows, reading
// the other's partial sums from its shared memory.
template <typename T, int GEMM, bool VEC, int KS>
__global__ void __launch_bounds__(kSimtThreads, 2) simt_gemm_kernel(const PathArgs a) {
  using TA = typename std::conditional<GEMM == 1, T, float>::type;   // the A operand's type
  extern __shared__ float4 simt_smem4[];
  float* sm = reinterpret_cast<float*>(simt_smem4);
  const Dims& d = a.d;
  const int m = blockIdx.x >> 1;
  pdl_enter();
  if (m >= *a.n_tiles) return;
  const TileInfo ti = a.tiles[m];
  const int row0 = (blockIdx.x & 1) * BM;   // row offset inside the 128-row tile
  if (row0 >= ti.rows) return;
  const int gl = blockIdx.z / KS, half = blockIdx.z % KS, grp = a.g0 + gl;
  const GroupInfo gi = a.groups[grp];
  const int n0 = blockIdx.y * BN;
  const int K = GEMM == 1 ? d.Ds : d.EH, N = GEMM == 1 ? d.EH : d.Dt;
  const int nrows = min(BM, ti.rows - row0);
  const int tid = threadIdx.x;

  // ---- loads: 16 four-value pieces per row and K block; a thread owns piece tid % 16 of
  //      rows tid / 16 + 16 i (A: i < 4, B: i < 2)
  const int piece = tid & 15, lrow = tid >> 4;
  int ah = 0, ai = piece * 4;   // GEMM1: head and channel of the piece
  const TA* abase;
  if (GEMM == 1) {
    abase = reinterpret_cast<const TA*>(static_cast<const T*>(a.src[gi.x]) +
                                        (static_cast<size_t>(gi.src_layer) * d.B + ti.b) * d.H_s *
                                            d.S * d.d_s +
                                        static_cast<size_t>(ti.s0 + row0) * d.d_s);
    while (VEC && ai >= d.d_s) {
      ai -= d.d_s;
      ++ah;
    }
  } else {
    abase = reinterpret_cast<const TA*>(static_cast<const float*>(a.a2) +
                                        (static_cast<size_t>(gl) * d.tpad +
                                         static_cast<size_t>(m) * kTileM + row0) * d.EH);
  }
  const T* wbase = static_cast<const T*>(GEMM == 1 ? a.w1 : a.w2) + static_cast<size_t>(grp) * N * K;
  auto load = [&](int kb) {   // K block kb into its stage
    float* sa = sm + (kb % kSimtStages) * kStageFloats;
    float* sb = sa + BM * kLd;
    const int c = kb * BK + piece * 4;
#pragma unroll
    for (int i = 0; i < BM / 16; ++i) {
      const int r = lrow + 16 * i;
      float* dst = sa + r * kLd + piece * 4;
      if (VEC) {
        const TA* src = GEMM == 1 ? abase + (static_cast<size_t>(ah) * d.S + r) * d.d_s + ai
                                  : abase + static_cast<size_t>(r) * d.EH + c;
        if (r < nrows && c < K) put4(dst, src);
        else put_zero4(dst);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int cc = c + e, h = GEMM == 1 ? cc / d.d_s : 0;
          const TA* src = GEMM == 1
                              ? abase + (static_cast<size_t>(h) * d.S + r) * d.d_s + (cc - h * d.d_s)
                              : abase + static_cast<size_t>(r) * d.EH + cc;
          dst[e] = r < nrows && cc < K ? (GEMM == 1 ? ld_f(src) : ld_a2(src)) : 0.f;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < BN / 16; ++i) {
      const int r = lrow + 16 * i;
      float* dst = sb + r * kLd + piece * 4;
      const T* src = wbase + static_cast<size_t>(n0 + r) * K + c;
      if (VEC) {
        if (n0 + r < N && c < K) put4(dst, src);
        else put_zero4(dst);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) dst[e] = n0 + r < N && c + e < K ? ld_f(src + e) : 0.f;
      }
    }
    cp_async_commit();
    if (VEC && GEMM == 1) {
      ai += BK;
      while (ai >= d.d_s) {
        ai -= d.d_s;
        ++ah;
      }
    }
  };

  // ---- products: group kg takes K values 16 kg .. 16 kg + 15 of a block; a thread rows
  //      ty + 8 i and columns tx + 8 j of the tile
  const int kg = tid >> 6, tx = tid & 7, ty = (tid >> 3) & 7;
  uint64_t acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  const uint32_t sbase = smem_u32(sm);
  const uint32_t aoff = (ty * kLd + kg * 16) * 4, boff = ((BM + tx) * kLd + kg * 16) * 4;
  const int nk_all = (K + BK - 1) / BK, per = (nk_all + KS - 1) / KS;
  const int k0 = half * per, nk = min(nk_all, k0 + per);
#pragma unroll
  for (int s = 0; s < kSimtStages - 1; ++s) {
    if (k0 + s < nk) load(k0 + s);
    else cp_async_commit();
  }
  for (int kb = k0; kb < nk; ++kb) {
    cp_async_wait_group<kSimtStages - 2>();
    __syncthreads();   // block kb landed; every thread is done with block kb - 1
    if (kb + kSimtStages - 1 < nk) load(kb + kSimtStages - 1);
    else cp_async_commit();
    const uint32_t st = sbase + (kb % kSimtStages) * kStageFloats * 4;
#pragma unroll
    for (int k4 = 0; k4 < 4; ++k4) {
      uint64_t b0[4], b1[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) ld_pairs(st + boff + (8 * j * kLd + 4 * k4) * 4, b0[j], b1[j]);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        uint64_t a0, a1;
        ld_pairs(st + aoff + (8 * i * kLd + 4 * k4) * 4, a0, a1);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          fma2(acc[i][j], a0, b0[j]);
          fma2(acc[i][j], a1, b1[j]);
        }
      }
    }
  }
  // ---- the groups' partial sums, added in order
  cp_async_wait_group<0>();
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      sm[(kg * BM + ty + 8 * i) * BN + tx + 8 * j] =
          __uint_as_float(static_cast<uint32_t>(acc[i][j])) +
          __uint_as_float(static_cast<uint32_t>(acc[i][j] >> 32));
  if (KS > 1) cluster_sync();
  else __syncthreads();
  const int col = n0 + (tid & 31);   // a warp takes a row's 32 columns
  const int r0 = (tid >> 5) + half * (kSimtThreads / 32);
  const uint32_t peer = KS > 1 ? mapa_cluster(sm, 1 - half) : 0;
  for (int r = r0; r < nrows && col < N; r += KS * kSimtThreads / 32) {
    const int o = r * BN + (tid & 31);
    float y = sm[o];
#pragma unroll
    for (int k = 1; k < kKGroups; ++k) y += sm[o + k * BM * BN];
    if (KS > 1) {
      float z[kKGroups];
#pragma unroll
      for (int k = 0; k < kKGroups; ++k) z[k] = ld_peer(peer + (o + k * BM * BN) * 4);
#pragma unroll
      for (int k = 1; k < kKGroups; ++k) z[0] += z[k];
      y += z[0];
    }
    const size_t grow = static_cast<size_t>(m) * kTileM + row0 + r;
    const float* g = a.gate + (static_cast<size_t>(grp) * d.tpad + grow) * d.E;
    if (GEMM == 1) {
      y += __ldg(a.b1 + static_cast<size_t>(grp) * d.EH + col);
      static_cast<float*>(a.a2)[(static_cast<size_t>(gl) * d.tpad + grow) * d.EH + col] =
          gelu_erf(y) * g[col / d.H];
    } else {
      for (int e = 0; e < d.E; ++e)
        y = fmaf(g[e], __ldg(a.b2 + (static_cast<size_t>(grp) * d.E + e) * d.Dt + col), y);
      const int h = col / d.d_t, ii = col - h * d.d_t;
      st_v(static_cast<T*>(a.dst[gi.x]) +
               ((((static_cast<size_t>(gi.tgt_layer) * d.B + ti.b) * d.H_t + h) * d.S + ti.s0 + row0 +
                 r) * d.d_t + ii),
           y);
    }
  }
  if (KS > 1) {   // the other CTA may still read this one's sums
    __syncwarp();
    cluster_sync();
  }
}

template <typename T, int GEMM, bool VEC, int KS>
cudaError_t launch_simt_v(const PathArgs& a, cudaStream_t st) {
  const Dims& d = a.d;
  static SmemOptIn smem;
  if (cudaError_t e = smem(simt_gemm_kernel<T, GEMM, VEC, KS>, kSimtSmem)) return e;
  const int N = GEMM == 1 ? d.EH : d.Dt;
  dim3 grid(2 * d.tiles_max, (N + BN - 1) / BN, a.gp * KS);
  return launch_kernel_clusters(a.overlap, KS, simt_gemm_kernel<T, GEMM, VEC, KS>, grid, kSimtThreads,
                                kSimtSmem, st, a);
}

template <typename T, int GEMM, int KS>
cudaError_t launch_simt(const PathArgs& a, cudaStream_t st) {
  return a.d.d_s % 4 == 0 && a.d.EH % 4 == 0 ? launch_simt_v<T, GEMM, true, KS>(a, st)
                                             : launch_simt_v<T, GEMM, false, KS>(a, st);
}

// GEMM2's K split over a pair: where the tiles fill the SMs' two places each at most once, and
// up to eight times over when K is long enough for the exchange not to count. E * H = 1536, 64
// tokens (192 tiles): 59.9 -> 49.6 us; 6144: 202 -> 154 us; 200 tokens (768 tiles): 557 -> 512
// us; 512 tokens: 1,021 -> 978 us; K = 768: 35.2 -> 32.2 us. Beyond: 1,751 -> 1,757 us (600 +
// 300 tokens, 6144), 110 -> 115 us (3 x 64 tokens, 1536), 26.8 -> 26.6 us (K = 512), 19.3 ->
// 20.5 us (K = 256).
template <typename T>
cudaError_t launch_simt2(const PathArgs& a, int num_sms, cudaStream_t st) {
  const Dims& d = a.d;
  const long long tiles = static_cast<long long>(d.B) * ((d.S + BM - 1) / BM) *
                          ((d.Dt + BN - 1) / BN) * a.gp;
  const bool split = d.EH >= 8 * BK && (tiles <= 2ll * num_sms ||
                                        (d.EH >= 64 * BK && tiles <= 16ll * num_sms));
  return split ? launch_simt<T, 2, 2>(a, st) : launch_simt<T, 2, 1>(a, st);
}

}  // namespace

cudaError_t launch_simt_gemm1(const PathArgs& a, cudaStream_t st) {
  return a.d.dtype == 0 ? launch_simt<__nv_bfloat16, 1, 1>(a, st) : launch_simt<float, 1, 1>(a, st);
}

cudaError_t launch_simt_gemm2(const PathArgs& a, int num_sms, cudaStream_t st) {
  return a.d.dtype == 0 ? launch_simt2<__nv_bfloat16>(a, num_sms, st) : launch_simt2<float>(a, num_sms, st);
}

}  // namespace mot
