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
// at 128 FMA per SM and clock, on 384 and 192 CTAs; the 16-byte reads take the load path for
// 1.5 times the FMAs' cycles, and the second GEMM's CTAs fill 1.3 waves. Measured there: 160
// and 209 us as 64 x 64 tiles of 4 x 4 threads (two scalar-fed reads per 16 FMAs, half of the
// SMs idle), 49 and 59 us so; 8 x 8 outputs a thread take 55 and 67 us with packed pairs (one
// CTA per SM) and 54 and 58 us with single FMAs.
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

// GEMM 1 or 2. Grid (2 * tiles_max, columns / 32, gp): blockIdx.x is a 64-row half tile.
// VEC: d_s and both K lengths are multiples of four, so every four-value piece is aligned and
// inside one row and head; otherwise values are read one by one.
template <typename T, int GEMM, bool VEC>
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
  const int gl = blockIdx.z, grp = a.g0 + gl;
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
#pragma unroll 1
        for (int e = 0; e < 4; ++e) {
          const int cc = c + e, h = GEMM == 1 ? cc / d.d_s : 0;
          const TA* src = GEMM == 1
                              ? abase + (static_cast<size_t>(h) * d.S + r) * d.d_s + (cc - h * d.d_s)
                              : abase + static_cast<size_t>(r) * d.EH + cc;
          dst[e] = r < nrows && cc < K ? ld_f(src) : 0.f;
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
#pragma unroll 1
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
  const int nk = (K + BK - 1) / BK;
#pragma unroll
  for (int s = 0; s < kSimtStages - 1; ++s) {
    if (s < nk) load(s);
    else cp_async_commit();
  }
  for (int kb = 0; kb < nk; ++kb) {
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
  __syncthreads();
  const int col = n0 + (tid & 31);   // a warp takes a row's 32 columns
  if (col >= N) return;
  for (int r = tid >> 5; r < nrows; r += kSimtThreads / 32) {
    const float* p = sm + r * BN + (tid & 31);
    float y = p[0];
#pragma unroll
    for (int k = 1; k < kKGroups; ++k) y += p[k * BM * BN];
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
}

template <typename T, int GEMM, bool VEC>
cudaError_t launch_simt_v(const PathArgs& a, cudaStream_t st) {
  const Dims& d = a.d;
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(simt_gemm_kernel<T, GEMM, VEC>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kSimtSmem);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const int N = GEMM == 1 ? d.EH : d.Dt;
  dim3 grid(2 * d.tiles_max, (N + BN - 1) / BN, a.gp);
  return launch_kernel(a.overlap, simt_gemm_kernel<T, GEMM, VEC>, grid, kSimtThreads, kSimtSmem, st, a);
}

template <typename T, int GEMM>
cudaError_t launch_simt(const PathArgs& a, cudaStream_t st) {
  return a.d.d_s % 4 == 0 && a.d.EH % 4 == 0 ? launch_simt_v<T, GEMM, true>(a, st)
                                             : launch_simt_v<T, GEMM, false>(a, st);
}

}  // namespace

cudaError_t launch_simt_gemm1(const PathArgs& a, cudaStream_t st) {
  return a.d.dtype == 0 ? launch_simt<__nv_bfloat16, 1>(a, st) : launch_simt<float, 1>(a, st);
}

cudaError_t launch_simt_gemm2(const PathArgs& a, cudaStream_t st) {
  return a.d.dtype == 0 ? launch_simt<__nv_bfloat16, 2>(a, st) : launch_simt<float, 2>(a, st);
}

}  // namespace mot
