// The recurrent scan of the backbone translators (App. C.2) in one launch on sm_103a:
// every slot of the window for a tile of tokens, from the source rows to the state h_r,
// without leaving the SM (the stages one by one are in bt.cu).
//
// One persistent CTA per SM walks (group, row tile) items; a tile holds whole tokens (tau x P
// of its 128 rows). Per slot, as in bt.cu: z = GELU(W_in LN_in(x) + b_in), q from LN_Q(h),
// k | v from LN_C(z), attention over the token's P rows, h += W_O o + b_O, h += FFN(LN_F(h)).
// The fp32 state lives in 128 columns of tensor memory for the whole scan; the residual sums, the
// layer norms and the attention are fp32 in the order of the staged kernels, and rows between the
// products are bf16 tiles in shared memory, rounded where those round them: the outputs agree bit
// for bit.
//
//   warps 0..7   epilogues, two per TMEM lane quarter: a thread owns 64 of a row's 128
//                columns; layer-norm statistics of the halves meet in shared memory.
//                Attention on packed fp32: a thread takes one head of two rows of a token.
//   warp 8       TMA producer: each slot's fp32 vectors, and the weights as 128 x 64 blocks
//                in the order of the products, through a ring that runs ahead over slots
//                and tiles.
//   warp 9       MMA issuer (M = 128, N = 128); warps 10 and 11 complete the warpgroup.
// Epilogues and products alternate through two mbarriers each way (go: operand tiles written,
// done: accumulators complete); the FFN keeps one 128-column chunk of products ahead.
// All waits are bounded; the epilogue warps agree on each, so they leave together.
//
// What bounds it: the epilogues and the waits between them; a tile's slot takes about 44,000
// cycles with 12 heads, of which 8,400 in the FFN's GELUs, 10,500 in the attention (6,000 with 2
// heads), 13,000 in the other epilogues' arithmetic and 12,000 waiting for products or for the
// slowest warp (the tensor cores work 7,000). The stages one by one move about 2.2 KB per row and
// slot through memory in 8 launches a slot; here a slot reads its 128-byte source rows and writes
// its 256-byte state rows. Measured, the translation as a whole: 8 x 1024 tokens of 12 heads, Top-1
// of 2, 4 slots: 2,778 us by staged kernels, 1,075 us; 7,923 ragged tokens of 2 heads, 8 slots:
// 1,362 and 376 us. Steps on the first: attention by one thread per row half, its loops over the
// keys unrolled, 168 registers and 0.5 to 1 KB of spills a thread 1,660; scores in tensor memory and
// the keys in loops 1,389; registers moved to the epilogue warpgroups (no spills) 1,279; two rows a
// thread 1,214; loops kept rolled and one call site for each role's wait and copy (the code of a
// slot, 183 KB, shrinks to 131 KB) 1,064; one row a thread for heads of 64 (their spills) 1,075.
// Attention on mma.sync with split bf16 weights and products summed in the state's own
// accumulators took 987 us, but moved outputs by 2e-3 of their norm through other roundings.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "bt_common.cuh"
#include "gelu.cuh"

namespace mot {
namespace {

constexpr int kScD = 128;                     // row width d
constexpr int kScEpi = 8;                     // epilogue warps
constexpr int kScThreads = 32 * (kScEpi + 4);  // three warpgroups: two epilogues, one of roles
// Registers a thread, per warpgroup: the launch's 168 (65,536 / 384, in eights) moved from the role
// warps to the epilogues, whose rows of 64 fp32 values and attention would spill.
constexpr int kScLaunchRegs = 168, kScEpiRegs = 216, kScRoleRegs = 72;
static_assert(2 * kScEpiRegs + kScRoleRegs <= 3 * kScLaunchRegs, "registers of the launch");
constexpr int kScBlk = 128 * 128;             // 128 rows x 64 bf16: a weight block, half a row tile
constexpr int kScTile = 2 * kScBlk;           // 128 rows x 128 bf16
constexpr int kScXch = 2 * 2 * 128 * 8;       // [parity][column half][row] (mean, M2)
constexpr int kScMaxRing = 7, kScMinRing = 4; // weight blocks in flight, as many as fit
// Shared memory: three row tiles, the exchange, barriers, two slots' vectors,
// the ring.
constexpr int kScOffXch = 3 * kScTile;
constexpr int kScOffBars = kScOffXch + kScXch;
constexpr int kScOffPrm = kScOffBars + 512;
constexpr int kScMaxSmem = 232448;

// One slot's fp32 vectors, contiguous (bt_scan_prm_floats): places of each.
enum PrmAt : int {
  kPrmSIn = 0, kPrmCIn = 128, kPrmLnC = 256, kPrmLnQ = 512, kPrmCQ = 768, kPrmCKv = 896,
  kPrmCO = 1152, kPrmLnF = 1280, kPrmCF2 = 1536, kPrmLnQn = 1664, kPrmCF1 = 1920
};
__host__ __device__ constexpr int prm_floats(int df) { return kPrmCF1 + df; }
constexpr int ring_off(int df) { return (kScOffPrm + 2 * prm_floats(df) * 4 + 1023) / 1024 * 1024; }
constexpr int ring_blocks(int df) {
  const int n = (kScMaxSmem - 1024 - ring_off(df)) / kScBlk;
  return n < kScMaxRing ? n : kScMaxRing;
}

// Packed pairs of fp32.
__device__ __forceinline__ uint64_t pk(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpk(uint64_t p) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(p));
  return f;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// gelu_tanh of two values
__device__ __forceinline__ uint64_t gelu2(uint64_t u) {
  const uint64_t k0 = pk(0.7978845608028654f, 0.7978845608028654f);
  const uint64_t k1 = pk(0.7978845608028654f * 0.044715f, 0.7978845608028654f * 0.044715f);
  const float2 x = unpk(mul2(u, fma2(k1, mul2(u, u), k0)));
  const uint64_t hu = mul2(u, pk(0.5f, 0.5f));
  return fma2(hu, pk(tanh_approx(x.x), tanh_approx(x.y)), hu);
}
// Two pairs (four values) of a vector in shared memory.
__device__ __forceinline__ void ld_pairs(uint32_t addr, uint64_t& a, uint64_t& b) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
}

// Registers of the executing warpgroup's threads, lowered or raised (every warp of it calls).
template <int N>
__device__ __forceinline__ void reg_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void reg_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

// Barrier id over n threads (n a multiple of 32).
__device__ __forceinline__ void bar_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// A thread's 64 columns of a row, as 32 pairs: one 64-column block of a 128B-swizzled tile.
__device__ __forceinline__ void store_row64(uint32_t tile, int row, int cg, const uint64_t (&v)[32]) {
  const uint32_t base = tile + cg * kScBlk + row * 128;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 f = unpk(v[4 * c + k]);
      w[k] = pack2(f.x, f.y);
    }
    st_shared_v4(base + ((c ^ (row & 7)) << 4), w[0], w[1], w[2], w[3]);
  }
}

__device__ __forceinline__ void load_acc(uint32_t addr, uint64_t (&v)[32]) {
  uint32_t r[32], u[32];
  tmem_ld_32x32b_x32(addr, r);
  tmem_ld_32x32b_x32(addr + 32, u);
  tmem_ld_wait(r);
  tmem_ld_wait(u);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    v[k] = pk(__uint_as_float(r[2 * k]), __uint_as_float(r[2 * k + 1]));
    v[16 + k] = pk(__uint_as_float(u[2 * k]), __uint_as_float(u[2 * k + 1]));
  }
}

__device__ __forceinline__ void add_vec(uint64_t (&v)[32], uint32_t b) {
#pragma unroll
  for (int c = 0; c < 16; ++c) {
    uint64_t x, y;
    ld_pairs(b + 16 * c, x, y);
    v[2 * c] = add2(v[2 * c], x);
    v[2 * c + 1] = add2(v[2 * c + 1], y);
  }
}

// The state rows' half in tensor memory: read onto v, and written back.
__device__ __forceinline__ void add_state(uint32_t addr, uint64_t (&v)[32]) {
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    uint32_t u[32];
    tmem_ld_32x32b_x32(addr + 32 * hf, u);
    tmem_ld_wait(u);
#pragma unroll
    for (int k = 0; k < 16; ++k)
      v[16 * hf + k] = add2(v[16 * hf + k],
                            pk(__uint_as_float(u[2 * k]), __uint_as_float(u[2 * k + 1])));
  }
}
__device__ __forceinline__ void store_state(uint32_t addr, const uint64_t (&v)[32]) {
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    uint32_t u[32];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float2 f = unpk(v[16 * hf + k]);
      u[2 * k] = __float_as_uint(f.x);
      u[2 * k + 1] = __float_as_uint(f.y);
    }
    tmem_st_32x32b_x32(addr + 32 * hf, u);
  }
  tmem_st_wait();
}

__device__ __forceinline__ void unpack8(const uint4& x, float (&f)[8]) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    f[2 * k] = bf16_lo(w[k]);
    f[2 * k + 1] = bf16_hi(w[k]);
  }
}

// Eight 32-bit columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_st8(uint32_t addr, const float (&f)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr),
               "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]), "f"(f[4]), "f"(f[5]), "f"(f[6]), "f"(f[7])
               : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t addr, float (&f)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(f[0]), "=f"(f[1]), "=f"(f[2]), "=f"(f[3]), "=f"(f[4]), "=f"(f[5]), "=f"(f[6]), "=f"(f[7])
      : "r"(addr)
      : "memory");
}

// Attention of the tile's first n_tok tokens over their own P rows, in fp32 and in the order of
// bt_attn_kernel: each dot product over its columns in turn, expf of the scaled scores less their
// maximum, normalised weights, the values added key by key. A thread takes one head of two rows of
// a token (heads of 64: of one row), so that a key or value is unpacked once for both; four keys to
// a step, whose scores wait in tensor memory (32 columns at `scratch`, this thread's own), so that
// the steps are loops. The output replaces the query rows (bf16) in qt; kt and vt: keys and values.
template <int DH>
struct Attn {
  static constexpr int NA = kScD / DH, CH = DH / 8;   // heads; 16-byte pieces of one
  static constexpr int NR = DH <= 32 ? 2 : 1;         // rows of a thread
};
struct AttnTask {   // rows p and p + ceil(P / NR), if it has one, of a token (first row rb); the head's first piece
  int rb, r[2], blk, c0;
  bool two;         // the second row is another one than the first
};
// Lanes past the tile's last task repeat it: no lane reads query rows that another warp overwrites.
template <int DH>
__device__ __forceinline__ AttnTask attn_task(int task, int P, int tau) {
  using A = Attn<DH>;
  const int per = (P + A::NR - 1) / A::NR;
  task = min(task, tau * A::NA * per - 1);
  const int th = task / per, p0 = task - th * per;
  const int tok = th / A::NA, hd = th - tok * A::NA;
  const int rb = tok * P;
  const bool two = p0 + per < P;
  return {rb, {rb + p0, rb + p0 + (two ? per : 0)}, ((hd * A::CH) >> 3) * kScBlk, (hd * A::CH) & 7, two};
}
template <int DH>
__device__ __forceinline__ void attend(uint8_t* qt, const uint8_t* kt, const uint8_t* vt, uint32_t scratch,
                                       const AttnTask& first, int n_tok, int P, int tau) {
  constexpr int NA = Attn<DH>::NA, CH = Attn<DH>::CH, NR = Attn<DH>::NR;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float scale = rsqrtf(static_cast<float>(DH));
  const int n_task = n_tok * NA * ((P + NR - 1) / NR);
#pragma unroll 1
  for (int t0 = warp * 32; t0 < n_task; t0 += 32 * kScEpi) {
    const AttnTask t = t0 == warp * 32 ? first : attn_task<DH>(t0 + lane, P, tau);
    auto at = [&](int r, int c) { return t.blk + r * 128 + (((t.c0 + c) ^ (r & 7)) << 4); };
    auto piece = [&](const uint8_t* tile, int r, int c) {
      return *reinterpret_cast<const uint4*>(tile + at(r, c));
    };
    __syncwarp();
    float m[NR];
#pragma unroll
    for (int n = 0; n < NR; ++n) m[n] = -INFINITY;
    {
      uint64_t q[NR][DH];   // each value twice: two keys take the halves of packed fp32
#pragma unroll
      for (int n = 0; n < NR; ++n)
#pragma unroll
        for (int c = 0; c < CH; ++c) {
          float f[8];
          unpack8(piece(qt, t.r[n], c), f);
#pragma unroll
          for (int k = 0; k < 8; ++k) q[n][8 * c + k] = pk(f[k], f[k]);
        }
#pragma unroll 1
      for (int j0 = 0; j0 < P; j0 += 4) {
        uint64_t s[NR][2];   // keys j0 + 2 h and j0 + 2 h + 1
#pragma unroll
        for (int n = 0; n < NR; ++n) s[n][0] = s[n][1] = 0ull;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
          float f[4][8];
#pragma unroll
          for (int i = 0; i < 4; ++i) unpack8(piece(kt, t.rb + min(j0 + i, P - 1), c), f[i]);
#pragma unroll
          for (int k = 0; k < 8; ++k)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const uint64_t kk = pk(f[2 * h][k], f[2 * h + 1][k]);
#pragma unroll
              for (int n = 0; n < NR; ++n) s[n][h] = fma2(q[n][8 * c + k], kk, s[n][h]);
            }
        }
        float x[8];   // x[2 i + n]: key j0 + i, row n
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float2 y = unpk(s[n % NR][h]);
            x[4 * h + n] = y.x * scale;
            x[4 * h + 2 + n] = y.y * scale;
          }
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (j0 + i < P)
#pragma unroll
            for (int n = 0; n < NR; ++n) m[n] = fmaxf(m[n], x[2 * i + n]);
        tmem_st8(scratch + 2 * j0, x);
      }
    }
    tmem_st_wait();
    float inv[NR];
#pragma unroll
    for (int n = 0; n < NR; ++n) inv[n] = 0.f;   // the sums first
#pragma unroll 1
    for (int j0 = 0; j0 < P; j0 += 4) {
      float x[8];
      tmem_ld8(scratch + 2 * j0, x);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int n = 0; n < NR; ++n) {
          x[2 * i + n] = expf(x[2 * i + n] - m[n]);
          if (j0 + i < P) inv[n] += x[2 * i + n];
        }
      tmem_st8(scratch + 2 * j0, x);
    }
    tmem_st_wait();
    uint64_t o[NR][DH / 2];
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      inv[n] = 1.f / inv[n];
#pragma unroll
      for (int k = 0; k < DH / 2; ++k) o[n][k] = 0ull;
    }
#pragma unroll 1
    for (int j0 = 0; j0 < P; j0 += 4) {
      float x[8];
      tmem_ld8(scratch + 2 * j0, x);
      auto step = [&](auto whole) {   // four keys, or the last P - j0
#pragma unroll
        for (int c = 0; c < CH; ++c) {
          uint4 u[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            u[i] = piece(vt, t.rb + (decltype(whole)::value ? j0 + i : min(j0 + i, P - 1)), c);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (!decltype(whole)::value && j0 + i >= P) break;
            float f[8];
            unpack8(u[i], f);
#pragma unroll
            for (int n = 0; n < NR; ++n) {
              const float w = x[2 * i + n] * inv[n];
#pragma unroll
              for (int k = 0; k < 4; ++k)
                o[n][4 * c + k] = fma2(pk(w, w), pk(f[2 * k], f[2 * k + 1]), o[n][4 * c + k]);
            }
          }
        }
      };
      if (j0 + 4 <= P) step(std::true_type{});
      else step(std::false_type{});
    }
    if (t0 + lane < n_task) {
#pragma unroll
      for (int n = 0; n < NR; ++n) {
        if (n == 1 && !t.two) break;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
          uint32_t u[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float2 f = unpk(o[n][4 * c + k]);
            u[k] = pack2(f.x, f.y);
          }
          *reinterpret_cast<uint4*>(qt + at(t.r[n], c)) = make_uint4(u[0], u[1], u[2], u[3]);
        }
      }
    }
  }
}

// The products of a slot, in order; from kStF on those of the FFN.
enum Stage : int { kStIn = 0, kStQ, kStK, kStV, kStO, kStF };
struct FfnStage {
  bool first;   // W_F1 of hidden chunk hc, else W_F2 of it
  int hc;
};
// W_F1 of chunks 0 and 1, then W_F2 of a chunk and W_F1 two chunks on, in turn (2 n_hc products).
__device__ __forceinline__ FfnStage ffn_stage(int i, int n_hc) {
  if (i == 2 * n_hc - 1) return {false, n_hc - 1};
  if (i == 0 || (i & 1)) return {true, (i + 1) >> 1};
  return {false, (i >> 1) - 1};
}

// NXV: 16-byte pieces of a source row per thread (d_s / 16); DH: attention head width.
template <int NXV, int DH>
__global__ void __launch_bounds__(kScThreads, 1)
    bt_scan_kernel(const __grid_constant__ CUtensorMap tmWin, const __grid_constant__ CUtensorMap tmWq,
                   const __grid_constant__ CUtensorMap tmWkv, const __grid_constant__ CUtensorMap tmWo,
                   const __grid_constant__ CUtensorMap tmWf1, const __grid_constant__ CUtensorMap tmWf2,
                   const BtArgs a, const GemmCfg c, const int n_ring, const int ring_at) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t sXQ = smem_u32(smem);        // LN_Q rows, q, attention output, LN_F rows
  const uint32_t sXZ = sXQ + kScTile;         // LN_C rows, v, hidden chunks 0, state rows out
  const uint32_t sKB = sXQ + 2 * kScTile;     // source rows, k, hidden chunks 1
  uint8_t* sRing = smem + ring_at;
  const uint32_t sPrm = smem_u32(smem + kScOffPrm);
  float2* xch = reinterpret_cast<float2*>(smem + kScOffXch);
  uint64_t* wfull = reinterpret_cast<uint64_t*>(smem + kScOffBars);   // [ring]
  uint64_t* wempty = wfull + kScMaxRing;
  uint64_t* pfull = wempty + kScMaxRing;   // [2] a slot's vectors landed
  uint64_t* pempty = pfull + 2;            // [2] read by every epilogue warp
  uint64_t* go = pempty + 2;           // [2] operand tiles written (every epilogue warp)
  uint64_t* done = go + 2;             // [2] accumulators complete
  uint64_t* drain = done + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const BtDims& d = a.d;
  constexpr int D = kScD, DS = 16 * NXV;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_hc = d.df / 128;
  const int total = total_items(a, c);
  const long long wl = a.wait_limit;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kScMaxRing; ++s) {
      mbar_init(&wfull[s], 1);
      mbar_init(&wempty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&pfull[i], 1);
      mbar_init(&pempty[i], kScEpi);
      mbar_init(&go[i], kScEpi);
      mbar_init(&done[i], 1);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kScEpi + 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const int prm_bytes = prm_floats(d.df) * 4;
  const uint32_t tmem = *tmem_slot;   // h at 0, accumulators at 128, 256 and 384
  uint32_t issued_mask = 0, issue_parity = 0, prm_issued = 0, prm_parity = 0;
  bool mma_issued = false;

  if (warp >= kScEpi) {
    reg_dec<kScRoleRegs>();   // the role warpgroup, its two idle warps included
    if (warp == kScEpi) {
      if (lane == 0) {
        // ------------------------------------------------ weights
        int slot = 0;
        uint32_t phase = 0, n_prm = 0;
        bool ok = true;
        auto put = [&](const CUtensorMap* map, int k0, int row) {
          if (!ok) return;
          if (!mbar_wait(&wempty[slot], phase ^ 1u, abort_flag, wl)) {
            ok = false;
            return;
          }
          mbar_arrive_expect_tx(&wfull[slot], kScBlk);
          tma_load_2d(sRing + slot * kScBlk, map, &wfull[slot], k0, row);
          issued_mask |= 1u << slot;
          issue_parity = (issue_parity & ~(1u << slot)) | (phase << slot);
          if (++slot == n_ring) {
            slot = 0;
            phase ^= 1u;
          }
        };
        for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
          const Work w = decode(a, c, it);
          if (!w.active) continue;
#pragma unroll 1
          for (int r = 0; r < d.N && ok; ++r) {
            const int gr = w.g * d.N + r;
            if (!mbar_wait(&pempty[n_prm & 1], ((n_prm >> 1) & 1) ^ 1u, abort_flag, wl)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(&pfull[n_prm & 1], prm_bytes);
            bulk_load(sPrm + (n_prm & 1) * prm_bytes, a.prm + int64_t(gr) * prm_floats(d.df), prm_bytes,
                      &pfull[n_prm & 1]);
            prm_issued |= 1u << (n_prm & 1);
            prm_parity = (prm_parity & ~(1u << (n_prm & 1))) | (((n_prm >> 1) & 1) << (n_prm & 1));
            ++n_prm;
#pragma unroll 1
            for (int st = 0; st < kStF + 2 * n_hc; ++st) {
              const CUtensorMap* map = st == kStIn ? &tmWin : st == kStQ ? &tmWq : st == kStO ? &tmWo : &tmWkv;
              int k0 = 0, row = st == kStIn ? w.g * D : st == kStK || st == kStV ? (2 * gr + st - kStK) * D : gr * D;
              if (st >= kStF) {
                const FfnStage f = ffn_stage(st - kStF, n_hc);
                map = f.first ? &tmWf1 : &tmWf2;
                if (f.first) row = gr * d.df + f.hc * 128;
                else k0 = f.hc * 128;
              }
#pragma unroll 1
              for (int kb = 0; kb < (st == kStIn ? 2 * DS / 64 : 2); ++kb) put(map, k0 + 64 * kb, row);
            }
          }
        }
      }
    } else if (warp == kScEpi + 1) {
      // ------------------------------------------------ MMA issuer (warp-uniform, elected lane)
      const uint32_t idesc = idesc_bf16_f32(128, 128);
      int slot = 0;
      uint32_t phase = 0, n_go = 0, n_done = 0;
      bool ok = true;
      for (int it = blockIdx.x; it < total && ok; it += gridDim.x) {
        const Work w = decode(a, c, it);
        if (!w.active) continue;
#pragma unroll 1
        for (int r = 0; r < d.N && ok; ++r) {
#pragma unroll 1
          for (int st = 0; st < kStF + 2 * n_hc && ok; ++st) {
            uint32_t acc = 128, tile = sXQ;
            bool go_first = false, commit = true, onto = false;
            switch (st) {
              case kStIn: tile = sKB; go_first = true; break;   // hi, then lo, x source rows
              case kStQ: acc = 256; go_first = r == 0; commit = false; break;   // r > 0: rows of the slot before
              case kStK: acc = 384; tile = sXZ; go_first = r > 0; break;
              case kStV: tile = sXZ; break;
              case kStO: go_first = true; break;
              default: {
                const FfnStage f = ffn_stage(st - kStF, n_hc);
                if (f.first) {
                  acc = 128 + 128 * (f.hc & 1);
                  go_first = f.hc == 0;
                } else {
                  acc = 384;
                  tile = (f.hc & 1) ? sKB : sXZ;
                  go_first = true;
                  commit = f.hc == n_hc - 1;
                  onto = f.hc > 0;
                }
              }
            }
            if (go_first) {
              if (!mbar_wait(&go[n_go & 1], (n_go >> 1) & 1, abort_flag, wl)) ok = false;
              ++n_go;
              tc_fence_after();
            }
            const int nblk = st == kStIn ? DS / 64 : 2, units = st == kStIn ? 2 * DS / 64 : 2;
            // `units` weight blocks against the A tile's 64-column blocks (1 or 2 of them, in turn)
#pragma unroll 1
            for (int u = 0; u < units && ok; ++u) {
              if (!mbar_wait(&wfull[slot], phase, abort_flag, wl)) {
                ok = false;
                break;
              }
              tc_fence_after();
              const uint64_t ad = sdesc_k_sw128(tile + (u & (nblk - 1)) * kScBlk);
              const uint64_t bd = sdesc_k_sw128(smem_u32(sRing + slot * kScBlk));
              if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                  umma_bf16(tmem + acc, ad + 2 * k, bd + 2 * k, idesc, onto || (u | k) != 0);
                umma_commit(&wempty[slot]);
              }
              __syncwarp();
              mma_issued = true;
              if (++slot == n_ring) {
                slot = 0;
                phase ^= 1u;
              }
            }
            if (commit) {
              if (ok && elect_one()) umma_commit(&done[n_done & 1]);
              __syncwarp();
              ++n_done;
            }
          }
        }
      }
    }
  } else {
    reg_inc<kScEpiRegs>();
    // ------------------------------------------------ epilogues
    const int q = warp & 3, cg = warp >> 2;
    const int row = q * 32 + lane;
    const int col0 = 64 * cg;
    const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
    const int t = row / d.P, p = row - t * d.P;
    const AttnTask task = attn_task<DH>(threadIdx.x, d.P, d.tau);
    uint32_t n_go = 0, n_done = 0, n_prm = 0, xpar = 0;
    bool ok = true;
    auto ready = [&]() {   // this warp's operand rows are written, its accumulator reads are done
      tc_fence_before();
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&go[n_go & 1]);
      ++n_go;
    };
    auto wait_done = [&]() -> bool {
      int wv = 1;
      if (lane == 0) wv = mbar_wait(&done[n_done & 1], (n_done >> 1) & 1, abort_flag, wl) ? 1 : 0;
      ++n_done;
      if (*abort_flag) wv = 0;
      ok = epi_and(1, 32 * kScEpi, __shfl_sync(0xffffffffu, wv, 0) != 0);
      tc_fence_after();
      return ok;
    };
    // statistics of a row of 2 n values, n in each of its two threads
    auto combine = [&](float n, float& mean, float& m2) {
      float2* x = xch + xpar * 256;
      xpar ^= 1u;
      x[cg * 128 + row] = make_float2(mean, m2);
      bar_sync(2 + q, 64);
      const float2 o = x[(cg ^ 1) * 128 + row];
      const float e = o.x - mean;
      m2 = (m2 + o.y) + e * e * (0.5f * n);
      mean = 0.5f * (mean + o.x);
    };
    // sums in column order, as row_stats of bt.cu
    auto stats = [&](const uint64_t (&v)[32], float& mean, float& m2) {
      float sum = 0.f;
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const float2 f = unpk(v[k]);
        sum += f.x;
        sum += f.y;
      }
      mean = sum * (1.f / 64);
      const uint64_t nm = pk(-mean, -mean);
      m2 = 0.f;
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const float2 f = unpk(add2(v[k], nm));
        m2 = fmaf(f.x, f.x, m2);
        m2 = fmaf(f.y, f.y, m2);
      }
      combine(64.f, mean, m2);
    };
    // tile <- bf16(gamma (v - mean) rstd + beta)
    auto store_ln = [&](uint32_t tile, const uint64_t (&v)[32], float mean, float rstd, uint32_t gb) {
      const uint64_t nm = pk(-mean, -mean), rs = pk(rstd, rstd);
      const uint32_t base = tile + cg * kScBlk + row * 128;
      gb += col0 * 4;
#pragma unroll
      for (int c = 0; c < 8; ++c) {   // eight columns at a time
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          uint64_t g0, g1, b0, b1;
          ld_pairs(gb + (8 * c + 4 * k) * 4, g0, g1);
          ld_pairs(gb + (D + 8 * c + 4 * k) * 4, b0, b1);
          const float2 y0 = unpk(fma2(mul2(add2(v[4 * c + 2 * k], nm), rs), g0, b0));
          const float2 y1 = unpk(fma2(mul2(add2(v[4 * c + 2 * k + 1], nm), rs), g1, b1));
          w[2 * k] = pack2(y0.x, y0.y);
          w[2 * k + 1] = pack2(y1.x, y1.y);
        }
        st_shared_v4(base + ((c ^ (row & 7)) << 4), w[0], w[1], w[2], w[3]);
      }
    };
    // the next active item at or after `it`
    auto next_item = [&](int it, Work& w) -> int {
      for (; it < total; it += gridDim.x) {
        w = decode(a, c, it);
        if (w.active) break;
      }
      return it;
    };
    // valid rows of a tile (its real tokens are a prefix), and this thread's half of its
    // source row in layer 0 (null: outside them)
    auto valid_rows = [&](const Work& w) -> int {
      const int n = a.routed ? w.ntok : min(w.ntok, seq_len_of(a, w.b) - w.s0);
      return n * d.P;
    };
    auto source = [&](const Work& w) -> const uint4* {
      if (row >= valid_rows(w)) return nullptr;
      int b = w.b, s = w.s0 + t;
      if (a.routed) {
        const int tok = __ldg(a.list + int64_t(w.g) * d.B * d.S + w.s0 + t);
        b = tok / d.S;
        s = tok - b * d.S;
      }
      return reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(a.src[w.g / d.E]) +
                                            ((int64_t(b) * d.P + p) * d.S + s) * DS + cg * (DS / 2));
    };
    // the state rows of the slot before, from sXZ: whole rows, a half warp each, this warp rows
    // 16 cg .. 16 cg + 15 of its quarter (written by this quarter's two warps)
    int64_t out_row = 0;
    int out_rows = 0;
    auto rows_out = [&]() {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int rr = q * 32 + cg * 16 + 2 * i + (lane >> 4), ch = lane & 15;
        if (rr < out_rows)
          reinterpret_cast<uint4*>(a.xo)[(out_row + rr) * (D / 8) + ch] =
              ld_shared_v4(sXZ + (ch >> 3) * kScBlk + rr * 128 + (((ch & 7) ^ (rr & 7)) << 4));
      }
      out_rows = 0;
      __syncwarp();
    };
    uint4 xv[NXV];
    auto load_x = [&](const uint4* src, int r) {
#pragma unroll
      for (int i = 0; i < NXV; ++i) xv[i] = make_uint4(0u, 0u, 0u, 0u);
      if (src != nullptr) {
        src += int64_t(a.src_layer[r]) * d.B * d.P * d.S * (DS / 8);
#pragma unroll
        for (int i = 0; i < NXV; ++i) xv[i] = __ldg(src + i);
      }
    };

    Work w;
    int it = next_item(blockIdx.x, w);
    const uint4* src = nullptr;
    if (it < total) load_x(src = source(w), 0);
    while (it < total && ok) {
      const int vrows = valid_rows(w), n_tok = vrows / d.P;
      const int64_t row0 = int64_t(w.g) * d.R + w.row0;   // the tile's first row (token-major)
      int it_n = it;
#pragma unroll 1
      for (int r = 0; r < d.N && ok; ++r) {
        // ---- source rows into the A tile, and their statistics
#pragma unroll
        for (int i = 0; i < NXV; ++i) {
          const int ch = cg * NXV + i;   // 16-byte piece of the row
          st_shared_v4(sKB + (ch >> 3) * kScBlk + row * 128 + (((ch & 7) ^ (row & 7)) << 4), xv[i].x,
                       xv[i].y, xv[i].z, xv[i].w);
        }
        ready();
        rows_out();   // while the product runs; the next write to sXZ comes after its wait
        bar_sync(2 + q, 64);   // both halves of the row are in the tile
        auto piece = [&](int ch) {
          return ld_shared_v4(sKB + (ch >> 3) * kScBlk + row * 128 + (((ch & 7) ^ (row & 7)) << 4));
        };
        float mu = 0.f, m2x = 0.f;
#pragma unroll
        for (int ch = 0; ch < 2 * NXV; ++ch) {
          const uint4 u = piece(ch);
          mu += bf16_lo(u.x) + bf16_hi(u.x) + bf16_lo(u.y) + bf16_hi(u.y) + bf16_lo(u.z) +
                bf16_hi(u.z) + bf16_lo(u.w) + bf16_hi(u.w);
        }
        mu *= 1.f / DS;
#pragma unroll
        for (int ch = 0; ch < 2 * NXV; ++ch) {
          const uint4 u = piece(ch);
          const uint32_t uw[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float lo = bf16_lo(uw[e]) - mu, hi = bf16_hi(uw[e]) - mu;
            m2x = fmaf(lo, lo, m2x);
            m2x = fmaf(hi, hi, m2x);
          }
        }
        const float rsx = rsqrtf(m2x * (1.f / DS) + kLnEps);
        // ---- z = GELU(LN-folded W_in x + c); LN_C(z); slot 0: h = z, LN_Q(h)
        if (lane == 0) mbar_wait(&pfull[n_prm & 1], (n_prm >> 1) & 1, abort_flag, wl);
        const uint32_t prm = sPrm + (n_prm & 1) * prm_bytes;
        uint64_t* prm_done = &pempty[n_prm & 1];
        ++n_prm;
        if (!wait_done()) break;   // agrees on both waits: a timed-out one sets the abort flag
        uint64_t v[32];
        float mean, m2;
        load_acc(tmem + lanes + 128 + col0, v);
        {
          const uint64_t nmu = pk(-mu, -mu), rs = pk(rsx, rsx);
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            uint64_t w0, w1, b0, b1;
            ld_pairs(prm + (kPrmSIn + col0) * 4 + 16 * k, w0, w1);
            ld_pairs(prm + (kPrmCIn + col0) * 4 + 16 * k, b0, b1);
            v[2 * k] = gelu2(fma2(fma2(nmu, w0, v[2 * k]), rs, b0));
            v[2 * k + 1] = gelu2(fma2(fma2(nmu, w1, v[2 * k + 1]), rs, b1));
          }
        }
        stats(v, mean, m2);
        {
          const float rstd = rsqrtf(m2 * (1.f / D) + kLnEps);
          store_ln(sXZ, v, mean, rstd, prm + kPrmLnC * 4);
          if (r == 0) {
            store_state(tmem + lanes + col0, v);
            store_ln(sXQ, v, mean, rstd, prm + kPrmLnQ * 4);
          }
        }
        ready();
        // ---- q, k, v rows
        if (!wait_done()) break;
        load_acc(tmem + lanes + 256 + col0, v);
        add_vec(v, prm + (kPrmCQ + col0) * 4);
        store_row64(sXQ, row, cg, v);
        load_acc(tmem + lanes + 384 + col0, v);
        add_vec(v, prm + (kPrmCKv + col0) * 4);
        store_row64(sKB, row, cg, v);
        if (!wait_done()) break;
        load_acc(tmem + lanes + 128 + col0, v);
        add_vec(v, prm + (kPrmCKv + D + col0) * 4);
        store_row64(sXZ, row, cg, v);
        bar_sync(1, 32 * kScEpi);
        // ---- attention over each token's rows
        attend<DH>(smem, smem + 2 * kScTile, smem + kScTile, tmem + lanes + 128 + col0, task,
                   n_tok, d.P, d.tau);
        ready();
        // ---- LN_F(h) of h += W_O o + b_O
        if (!wait_done()) break;
        load_acc(tmem + lanes + 128 + col0, v);
        add_vec(v, prm + (kPrmCO + col0) * 4);
        add_state(tmem + lanes + col0, v);
        store_state(tmem + lanes + col0, v);
        stats(v, mean, m2);
        store_ln(sXQ, v, mean, rsqrtf(m2 * (1.f / D) + kLnEps), prm + kPrmLnF * 4);
        ready();
        // the next slot's source rows (or the next tile's first), used after the FFN
        if (r + 1 < d.N) {
          load_x(src, r + 1);
        } else {
          it_n = next_item(it + gridDim.x, w);
          if (it_n < total) load_x(src = source(w), 0);
        }
        // ---- FFN hidden chunks
#pragma unroll 1
        for (int hc = 0; hc < n_hc; ++hc) {
          if (!wait_done()) break;
          load_acc(tmem + lanes + 128 + 128 * (hc & 1) + col0, v);
          add_vec(v, prm + (kPrmCF1 + hc * 128 + col0) * 4);
#pragma unroll
          for (int k = 0; k < 32; ++k) v[k] = gelu2(v[k]);
          store_row64((hc & 1) ? sKB : sXZ, row, cg, v);
          ready();
        }
        // ---- h_r: statistics for LN_out, rows out, LN_Q for the next slot
        if (!ok || !wait_done()) break;
        load_acc(tmem + lanes + 384 + col0, v);
        add_vec(v, prm + (kPrmCF2 + col0) * 4);
        add_state(tmem + lanes + col0, v);
        if (r + 1 < d.N) store_state(tmem + lanes + col0, v);
        store_row64(sXZ, row, cg, v);
        stats(v, mean, m2);   // its barrier covers this lane quarter's rows of sXZ too
        const int64_t slot_row = int64_t(r) * d.G * d.R;
        if (r + 1 < d.N)
          store_ln(sXQ, v, mean, rsqrtf(m2 * (1.f / D) + kLnEps), prm + kPrmLnQn * 4);
        __syncwarp();
        if (lane == 0) mbar_arrive(prm_done);   // this warp's last read of the slot's vectors
        if (row < vrows && cg == 0) a.rstat[slot_row + row0 + row] = make_float2(mean, m2);
        out_row = slot_row + row0;
        out_rows = vrows;
      }
      it = it_n;
    }
    if (ok) rows_out();
  }

  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // unwinding after a timed-out wait: let issued copies land and issued MMAs finish
    if (warp == kScEpi && lane == 0) {
      for (int s = 0; s < 2; ++s)
        if ((prm_issued >> s) & 1u) {
          const uint32_t ad = smem_u32(&pfull[s]);
          const long long t0 = clock64();
          while (!mbar_try_wait(ad, (prm_parity >> s) & 1u) && clock64() - t0 < wl) {
          }
        }
      for (int s = 0; s < n_ring; ++s)
        if ((issued_mask >> s) & 1u) {
          const uint32_t ad = smem_u32(&wfull[s]);
          const long long t0 = clock64();
          while (!mbar_try_wait(ad, (issue_parity >> s) & 1u) && clock64() - t0 < wl) {
          }
        }
    }
    if (warp == kScEpi + 1 && mma_issued) {
      if (elect_one()) umma_commit(drain);
      __syncwarp();
      const uint32_t ad = smem_u32(drain);
      const long long t0 = clock64();
      while (!mbar_try_wait(ad, 0) && clock64() - t0 < wl) {
      }
    }
    __syncthreads();
  }
  if (warp == kScEpi + 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (threadIdx.x == 0 && *abort_flag) atomicOr(a.status, kStatusTimeout);
}

template <int NXV, int DH>
cudaError_t launch_scan(const BtArgs& a, const CUtensorMap (&tm)[6], int num_sms, cudaStream_t st) {
  const BtDims& d = a.d;
  GemmCfg c{};
  c.mode = kBtIn;   // row tiles of whole tokens
  c.groups = d.G;
  c.row_tiles = d.B * d.tiles_b;
  c.n_tiles = 1;
  auto kern = bt_scan_kernel<NXV, DH>;
  static SmemOptIn smem;
  if (cudaError_t e = smem(kern, kScMaxSmem)) return e;
  const int n_ring = ring_blocks(d.df), at = ring_off(d.df);
  const long long items = static_cast<long long>(c.groups) * c.row_tiles;
  const int grid = static_cast<int>(items < num_sms ? items : num_sms);
  if (grid <= 0) return cudaSuccess;
  kern<<<grid, kScThreads, at + n_ring * kScBlk + 1024, st>>>(tm[0], tm[1], tm[2], tm[3], tm[4],
                                                              tm[5], a, c, n_ring, at);
  return cudaGetLastError();
}

}  // namespace

int bt_scan_prm_floats(const BtDims& d) { return prm_floats(d.df); }

// One slot's vectors of group g, from the load-time arrays ([g][..] or [g][slot][..]).
void bt_scan_pack_prm(const BtDims& d, const BtScanVecs& v, int g, int slot, float* out) {
  const size_t D = d.d, gr = size_t(g) * d.N + slot;
  auto put = [&](int at, const float* src, size_t n) { std::copy(src, src + n, out + at); };
  put(kPrmSIn, v.s_in + g * D, D);
  put(kPrmCIn, v.c_in + g * D, D);
  put(kPrmLnC, v.ln_c + gr * 2 * D, 2 * D);
  put(kPrmLnQ, v.ln_q + gr * 2 * D, 2 * D);
  put(kPrmCQ, v.c_q + gr * D, D);
  put(kPrmCKv, v.c_kv + gr * 2 * D, 2 * D);
  put(kPrmLnF, v.ln_f + gr * 2 * D, 2 * D);
  put(kPrmLnQn, v.ln_q + (slot + 1 < d.N ? gr + 1 : gr) * 2 * D, 2 * D);
  put(kPrmCF1, v.c_f1 + gr * d.df, d.df);
  put(kPrmCO, v.c_o + gr * D, D);
  put(kPrmCF2, v.c_f2 + gr * D, D);
}

// Rows of 128 (one 128-column tile of state), an FFN in whole 128-column chunks whose vectors
// leave room for the ring (d_f up to 4,096), and a window of at most 16 slots (the state
// rows of every slot are kept for the output projections).
bool bt_scan_supported(const BtDims& d) {
  return d.d == kScD && d.df % 128 == 0 && d.df <= 4096 && ring_blocks(d.df) >= kScMinRing &&
         d.N <= 16;
}

cudaError_t launch_bt_scan(const BtArgs& a, const CUtensorMap (&tm)[6], int num_sms,
                           cudaStream_t st) {
  const int dh = a.d.d / a.d.na;
  if (a.d.d_s == 64)
    return dh == 16   ? launch_scan<4, 16>(a, tm, num_sms, st)
           : dh == 32 ? launch_scan<4, 32>(a, tm, num_sms, st)
                      : launch_scan<4, 64>(a, tm, num_sms, st);
  return dh == 16   ? launch_scan<8, 16>(a, tm, num_sms, st)
         : dh == 32 ? launch_scan<8, 32>(a, tm, num_sms, st)
                    : launch_scan<8, 64>(a, tm, num_sms, st);
}

}  // namespace mot
