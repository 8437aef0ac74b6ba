// Attention of one replay layer over gathered key and value rows (App. C.4) on
// sm_103a: the source-guided layers (the Top-S rows of replay_select), and the full
// causal layers whose shapes the tcgen05 kernel (replay_fmha.cu) does not tile.
//
//   replay_gather_kernel  one item per (b, key/value head, u), one warp per item: all
//                         query heads of the GQA group attend to the same rows, so the
//                         warp computes S^T = K_rows Q^T and O^T = V_rows^T P^T on
//                         mma.m16n8k16 with the heads as its 8 columns. The rows reach
//                         the warp through its own ring of 4 KB tiles in shared memory,
//                         filled by cp.async three tiles ahead, across item boundaries,
//                         and are read by ldmatrix (the value tiles transposed). No
//                         warp waits for another: a tile is handed over by the warp's
//                         own copy groups.
//
// What bounds it: the gathers, S * 2 * d * 2 bytes per item out of L2 (2.15 GB for
// 4 x 4096 positions, 2 key/value heads, d = 128, S = 128; 15.6 TB/s, L2-to-SM links 54%
// busy on average and 64% on the busiest slice). Why warps on mma.sync and not the
// fifth-generation tensor cores: the products are small (heads x S x d), and a tcgen05
// item needs a lane of four warps with 72 KB of tiles, four barriers and two serial MMA
// round trips, so only three items are in flight per SM; here twelve are, each with 12 to
// 16 KB of copies outstanding and nothing to wait for but those. Measured at that size:
// 252 us as three tcgen05 lanes, 248 us with the MMA fragments loaded straight from global
// memory (each 16-byte load instruction touches 4 to 8 rows: 1,650 L1 wavefronts per item),
// 177 us with this ring and a general tile cursor (3,200 instructions per item), 162 us
// with the static tile stream (1,550), 142 to 151 us with the tile orders below, 140 us with the
// item order below and the selection's spare slots spread (pad_row in replay.cu).
//
// Probabilities that the CUDA-core kernel before this one held in fp32 (heads of 64, sets past
// 128 rows, full layers) stay fp32: three bf16 parts, exact. Two parts rounded to 2^-17 moved the
// error against 64 bits from 1.630332e-3 to 1.630333e-3; with three it is the
// former kernel's to eight digits, with the small parts added apart from the large one where they
// take MMAs of their own (three sums into one accumulator over 1,500 rows: + 2e-10). The time on
// CUDA cores, with two parts, and with three and today's order of items: 8 x 1024 positions, 12
// heads of 64, S = 128: 691, 213, 204 us; 4 x 4096, 12 heads of 128 on 2, S = 256: 1,127, 248, 279
// us; full causal layers of 2047 + 1025 positions, the same heads: 984, 232, 259 us.
#include "replay_common.cuh"

namespace mot {
namespace {

// How a probability enters the second product: as bf16; or as the sum of three bf16 (hi + mid +
// lo: its fp32, exactly), the parts of one or two heads in different columns (no extra MMA),
// of 3 or 4 heads two parts in columns and one in a second MMA, else in three MMAs.
enum ProbForm : int { kProbBf16 = 0, kProbCols1 = 1, kProbCols2 = 2, kProbCols4 = 4, kProbMma3 = 8 };

constexpr int kRgStages = 4;
constexpr int kRgTile = 4096;

// Shared memory: 12 warps of one 8-head column tile fill the SM (18 KB each); two column
// tiles double the accumulators, so 8 warps of up to 255 registers.
template <int D, int NT>
struct Rg {
  static constexpr int kWarps = NT == 1 ? 12 : 8;
  static constexpr int kRow = 2 * D;                    // bytes of a key or value row
  static constexpr int kRows = kRgTile / kRow;          // rows per tile: 16 or 32
  static constexpr int kLpr = kRow / 16;                // lanes (16-byte chunks) per row
  static constexpr int kQ = 8 * NT * kRow;              // query rows in, output rows out
  static constexpr int kWarpBytes = kRgStages * kRgTile + kQ;
  static constexpr int kSmem = kWarps * kWarpBytes + 1024;
};

__device__ __forceinline__ void stsm4_t(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2,
                                        uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr),
               "r"(r0), "r"(r1), "r"(r2), "r"(r3)
               : "memory");
}

// Transpose of the warp's 8 x 8 matrix of 16-bit values (row lane / 4, columns
// 2 (lane % 4) and + 1 in each register).
__device__ __forceinline__ uint32_t movm_t(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

__device__ __forceinline__ void prefetch_l1(const void* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// fp32 as three bf16 without rounding: the upper half of x holds 8 of its 24 significant bits, that of
// what is left below it (exact) the next 8 from its leading one, and what is below those fits in 8.
__device__ __forceinline__ float below_bf16(float x) {
  return x - __uint_as_float(__float_as_uint(x) & 0xFFFF0000u);
}
__device__ __forceinline__ uint32_t upper_halves(float x, float y) {
  return __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
}

// Two bf16 each: acc + 0 w, which is NaN from the first infinity or NaN on.
__device__ __forceinline__ uint32_t zero_times(uint32_t w, uint32_t acc) {
  uint32_t r;
  asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(w), "r"(0u), "r"(acc));
  return r;
}

// The values of an item that came out infinite or NaN, again: one warp, key by key in fp32. In the
// MMAs an infinite value row also meets the probability 0 of the slots that fill up a unit, and
// the small parts of its own probability, which may be 0: infinity times 0 is NaN. Here it meets
// its own probability alone. Everything finite stays.
template <int D>
__device__ __noinline__ void redo_non_finite(const ReplayArgs& a, int bh, int u, int n, const int32_t* sel) {
  constexpr int DL = D / 32;   // dimensions per lane
  const ReplayDims& d = a.d;
  const int lane = threadIdx.x & 31, G = d.Hq / d.Hkv;
  const float scale = rsqrtf(float(D));
  const uint16_t* kb = static_cast<const uint16_t*>(a.k) + int64_t(bh) * d.N * D;
  const uint16_t* vb = static_cast<const uint16_t*>(a.v) + int64_t(bh) * d.N * D;
  for (int h = 0; h < G; ++h) {
    const int64_t at = ((int64_t(bh) * G + h) * d.N + u) * D;
    const uint16_t* qr = static_cast<const uint16_t*>(a.q) + at;
    auto key = [&](int j) { return sel == nullptr ? j : sel[j]; };
    auto score = [&](int row) {
      const uint16_t* kr = kb + int64_t(row) * D;
      float x = 0.f;
#pragma unroll 1
      for (int c = 0; c < D; ++c) x = fmaf(bf16f(qr[c]) * scale, bf16f(kr[c]), x);
      return x;
    };
    float m = -INFINITY, l = 0.f, o[DL];
#pragma unroll 1
    for (int j = lane; j < n; j += 32) m = fmaxf(m, score(key(j)));
    for (int w = 16; w > 0; w >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, w));
#pragma unroll
    for (int e = 0; e < DL; ++e) o[e] = 0.f;
#pragma unroll 1
    for (int j0 = 0; j0 < n; j0 += 32) {
      const bool in = j0 + lane < n;
      const int row = in ? key(j0 + lane) : 0;
      const float p = in ? expf(score(row) - m) : 0.f;
      l += p;
#pragma unroll 1
      for (int i = 0; i < min(32, n - j0); ++i) {
        const float pi = __shfl_sync(0xffffffffu, p, i);
        const uint16_t* vr = vb + int64_t(__shfl_sync(0xffffffffu, row, i)) * D + lane * DL;
#pragma unroll
        for (int e = 0; e < DL; ++e) o[e] = fmaf(pi, bf16f(vr[e]), o[e]);
      }
    }
    for (int w = 16; w > 0; w >>= 1) l += __shfl_xor_sync(0xffffffffu, l, w);
    uint16_t* out = static_cast<uint16_t*>(a.out) + at + lane * DL;
#pragma unroll
    for (int e = 0; e < DL; ++e)
      if ((out[e] & 0x7F80u) == 0x7F80u) out[e] = __bfloat16_as_ushort(__float2bfloat16_rn(o[e] / l));
  }
}

// One unit of a warp's work: rows c0 .. c0 + CH - 1 of the set of one item
// (bh = b * Hkv + hk, position u); bh < 0 past the last item.
struct Unit {
  int bh, v, u, n, c0;   // v: step of the walk over the positions u; n: rows of the item's set
};

// D: head width; NT: 8-head column tiles; PF: ProbForm; CH: rows per unit; MULTI: sets of
// more than CH rows (online softmax over the units of an item); FULL: the set is 0 .. u.
//
// A unit is TPC key tiles, then the TPC value tiles of the same rows. While the warp
// multiplies tile i of this stream it copies tile i + 4, which is one of this unit or of the
// next; 2 TPC is a multiple of the ring's 4 stages, so every tile's stage, shared-memory
// address and successor are constants of the unrolled code. Slots past the end of a set
// repeat one of its rows (the selection pads its workspace rows) with probability 0.
template <int D, int NT, int PF, int CH, bool MULTI, bool FULL>
__global__ void __launch_bounds__(32 * Rg<D, NT>::kWarps, 1)
    replay_gather_kernel(const ReplayArgs a) {
  using C = Rg<D, NT>;
  constexpr int MT = CH / 16, DT = D / 16, TPC = CH / C::kRows, MPT = C::kRows / 16;
  static_assert(TPC >= 2 && (2 * TPC) % kRgStages == 0, "tile stream");
  extern __shared__ uint8_t smem_raw[];
  pdl_enter();
  const ReplayDims& d = a.d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int G = d.Hq / d.Hkv;
  if (a.stall_test && blockIdx.x == 0) {   // test hook for the report of a timeout: the kernel waits for
    // nothing but its own copies, so this is a bounded wait of the hook's own
    __shared__ uint64_t never;
    __shared__ int gave_up;
    if (threadIdx.x == 0) {
      gave_up = 0;
      mbar_init(&never, 1);
      fence_barrier_init();
      if (!mbar_wait(&never, 0, &gave_up, a.wait_limit)) atomicOr(a.status, kStatusTimeout);
    }
    return;
  }
  const uint32_t ring = ((smem_u32(smem_raw) + 1023u) & ~1023u) + warp * C::kWarpBytes;
  const uint32_t qbuf = ring + kRgStages * kRgTile;
  constexpr float sl2 = float((D == 64 ? 0.125 : 0.08838834764831844) * 1.4426950408889634);   // log2(e) / sqrt(d)

  // items v * n_bh + bh, from the warp's index on in steps of the grid's warps: the
  // warps at work spread over the heads, so their hot rows spread over the L2. With 16 positions or
  // more to a pass, a pass is whole positions (a few warps may idle) and a warp turns to the next
  // head with each: were it to stay with one sequence, the warps of a ragged batch's short ones
  // would stand idle (eight sequences of 4,096 to 100 positions, 28 heads on 4, S = 128: 391 us, 127
  // now; 2,500 + 700 positions, 12 heads on 2: 59 and 50).
  const int n_bh = d.B * d.Hkv;
  const int warps = static_cast<int>(gridDim.x) * C::kWarps;
  const bool turn = warps >= 16 * n_bh;
  const int step_v = warps / n_bh, step_bh = turn ? 1 : warps - step_v * n_bh;
  const int step = turn ? step_v * n_bh : warps;
  auto advance = [&](Unit& w) {
    w.bh += step_bh;
    w.v += step_v;
    if (w.bh >= n_bh) {
      w.bh -= n_bh;
      if (!turn) ++w.v;
    }
  };
  auto place = [&](Unit& w) { w.u = FULL ? d.N - 1 - w.v : w.v; };   // full: longest sets first
  auto settle = [&](Unit& w) {   // skip to an item inside its sequence
    place(w);
    while (w.v < d.N && w.u >= seq_len_of(a, w.bh / d.Hkv)) {
      advance(w);
      place(w);
    }
    w.c0 = 0;
    w.n = FULL ? w.u + 1 : min(d.S, w.u + 1);
    if (w.v >= d.N) w.bh = -1;
  };
  auto next_unit = [&](const Unit& w) {
    Unit x = w;
    if (MULTI && w.c0 + CH < w.n) {
      x.c0 += CH;
      return x;
    }
    advance(x);
    settle(x);
    return x;
  };
  // a CTA's warps start on neighbouring items (the key/value heads of a position share its
  // selection: 3% faster); with fewer items than warps they spread over the SMs instead
  const int nb = static_cast<int>(gridDim.x), blk = static_cast<int>(blockIdx.x);
  const int first = int64_t(n_bh) * d.N < step ? warp * nb + blk : blk * C::kWarps + warp;
  Unit cur;
  cur.v = first / n_bh;
  cur.bh = first - cur.v * n_bh;
  settle(cur);
  if (first >= step) cur.bh = -1;

  // ---- copies: a lane moves the 16-byte chunk `chunk` of rows 8 grp .. 8 grp + 7 of a tile
  const int grp = lane / C::kLpr, chunk = lane % C::kLpr;
  uint32_t dsto[8];   // swizzled place of the lane's chunk of row i, stage 0
#pragma unroll
  for (int i = 0; i < 8; ++i)
    dsto[i] = ring + grp * 8 * C::kRow + i * C::kRow + (((chunk & 7) ^ i) << 4) +
              ((chunk & ~7) << 4);
  auto sel_of = [&](const Unit& w) {
    return a.sel + (int64_t(w.bh / d.Hkv) * d.N + w.u) * a.sel_stride + w.c0 + 8 * grp;
  };
  // the warps of a CTA take the tiles of a set in different orders: neighbouring positions
  // share their most wanted rows, and reading those at the same moment queues at one L2 slice
  const int rot = FULL ? 0 : warp % TPC * C::kRows;
  // positions of the lane's rows of tile ti of unit w, read one tile before the copies use them
  int idx[8];
  auto load_idx = [&](const Unit& w, const int32_t* sel, int ti) {
    const int tr = ti % TPC;
    if (FULL) {
#pragma unroll
      for (int i = 0; i < 8; ++i) idx[i] = min(w.c0 + tr * C::kRows + 8 * grp + i, w.n - 1);
    } else if (w.bh >= 0) {
      const int off = (tr * C::kRows + rot) & (CH - 1);
      const int4 x = ld_chain(reinterpret_cast<const int4*>(sel + off));
      const int4 y = ld_chain(reinterpret_cast<const int4*>(sel + off + 4));
      idx[0] = x.x; idx[1] = x.y; idx[2] = x.z; idx[3] = x.w;
      idx[4] = y.x; idx[5] = y.y; idx[6] = y.z; idx[7] = y.w;
    }
  };
  // tile ti of unit w (keys for ti < TPC, else values) into its stage
  auto copy_tile = [&](const Unit& w, int ti) {
    if (w.bh >= 0) {
      const char* src = static_cast<const char*>(ti < TPC ? a.k : a.v) +
                        int64_t(w.bh) * d.N * C::kRow + chunk * 16;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        cp_async_16(dsto[i] + (ti % kRgStages) * kRgTile,
                    src + uint32_t(idx[i]) * uint32_t(C::kRow));
    }
    cp_async_commit();
  };

  // ---- queries: 16-byte pieces of the 8 NT columns' rows
  constexpr int QV = 8 * NT * C::kLpr / 32;   // per lane
  uint4 qn[QV];
  auto load_q = [&](const Unit& w) {
#pragma unroll
    for (int i = 0; i < QV; ++i) {
      const int e = i * 32 + lane, c = e % C::kLpr;
      int h = e / C::kLpr;
      if (PF == kProbCols1 || PF == kProbCols2 || PF == kProbCols4) h &= PF - 1;   // repeated heads
      qn[i] = make_uint4(0u, 0u, 0u, 0u);
      if (h < G)
        qn[i] = __ldg(reinterpret_cast<const uint4*>(
            static_cast<const uint16_t*>(a.q) +
            ((int64_t(w.bh) * G + h) * d.N + w.u) * D + 8 * c));
    }
  };
  // ldmatrix lane addresses: matrix mi = lane / 8, row r = lane % 8 of it. Chunk c of a row
  // sits at (c ^ (row % 8)) in its 128-byte half, so a step over chunk pairs is an XOR of
  // bits 5 and 6 and, past 128 bytes, an offset.
  const int mi = lane >> 3, r = lane & 7;
  uint32_t ka[4], va[4], qa[2];
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    ka[x] = (ring + (r + 8 * (mi & 1)) * C::kRow + (((mi >> 1) ^ r) << 4)) ^ (x << 5);
    va[x] = (ring + (r + 8 * (mi >> 1)) * C::kRow + (((mi & 1) ^ r) << 4)) ^ (x << 5);
  }
#pragma unroll
  for (int x = 0; x < 2; ++x) qa[x] = (qbuf + r * C::kRow + ((mi ^ r) << 4)) ^ (x << 6);

  const int32_t* sel_c = nullptr;
  if (cur.bh >= 0) {
    sel_c = sel_of(cur);
    load_q(cur);
  }
  Unit nxt = cur.bh >= 0 ? next_unit(cur) : cur;
  const int32_t* sel_n = nullptr;
  auto next_sel = [&]() {
    if (nxt.bh < 0) return;
    sel_n = sel_of(nxt);
    if (!FULL && lane < CH / 32) prefetch_l1(sel_n - 8 * grp + 32 * lane);
  };
  next_sel();
  load_idx(cur, sel_c, 0);
#pragma unroll
  for (int i = 0; i < kRgStages; ++i) {
    copy_tile(cur, i);
    if (i + 1 < 2 * TPC) load_idx(cur, sel_c, i + 1);
    else load_idx(nxt, sel_n, 0);
  }

  float o[NT][DT][4], l[NT][4], m[NT][2];
  uint32_t qf[NT][DT][2];
  while (cur.bh >= 0) {
    if (!MULTI || cur.c0 == 0) {
      // a new item: its queries, through the warp's buffer, into the MMA's column operand
      __syncwarp();
#pragma unroll
      for (int i = 0; i < QV; ++i) {
        const int e = i * 32 + lane, h = e / C::kLpr, c = e % C::kLpr;
        st_shared_v4(qbuf + h * C::kRow + ((((c & 7) ^ (h & 7)) | (c & ~7)) << 4), qn[i].x,
                     qn[i].y, qn[i].z, qn[i].w);
      }
      __syncwarp();
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int s2 = 0; s2 < DT / 2; ++s2) {   // chunks 4 s2 .. 4 s2 + 3: K steps 2 s2, 2 s2 + 1
          uint32_t x[4];
          ldsm4(qa[s2 & 1] + nt * 8 * C::kRow + (s2 >> 1) * 128, x);
          qf[nt][2 * s2][0] = x[0];
          qf[nt][2 * s2][1] = x[1];
          qf[nt][2 * s2 + 1][0] = x[2];
          qf[nt][2 * s2 + 1][1] = x[3];
        }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
        for (int i = 0; i < DT; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) o[nt][i][e] = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) l[nt][e] = 0.f;
        m[nt][0] = m[nt][1] = -INFINITY;
      }
    }
    auto copy_ahead = [&](int ti) {   // tile ti + 4 of the stream, into the stage of tile ti
      __syncwarp();
      constexpr int T = 2 * TPC;
      const int ahead = ti + kRgStages;
      if (ahead < T) copy_tile(cur, ahead);
      else copy_tile(nxt, ahead - T);
      if (ahead + 1 < T) load_idx(cur, sel_c, ahead + 1);
      else if (ahead + 1 < 2 * T) load_idx(nxt, sel_n, ahead + 1 - T);
    };
    // ---- S^T = K_rows Q^T (two accumulation chains per 16 rows)
    float s[NT][MT][4];
#pragma unroll
    for (int ti = 0; ti < TPC; ++ti) {
      cp_async_wait_group<kRgStages - 1>();
      __syncwarp();
      float acc[2][NT][MPT][4];
#pragma unroll
      for (int e = 0; e < 8 * NT * MPT; ++e) (&acc[0][0][0][0])[e] = 0.f;
#pragma unroll
      for (int st = 0; st < DT; ++st)
#pragma unroll
        for (int mk = 0; mk < MPT; ++mk) {
          uint32_t x[4];
          ldsm4(ka[st & 3] + (ti % kRgStages) * kRgTile + mk * 16 * C::kRow + (st >> 2) * 128, x);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
            mma_bf16(acc[st & 1][nt][mk], x[0], x[1], x[2], x[3], qf[nt][st][0], qf[nt][st][1]);
        }
      copy_ahead(ti);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int mk = 0; mk < MPT; ++mk)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            s[nt][ti * MPT + mk][e] = acc[0][nt][mk][e] + acc[1][nt][mk][e];
    }
    if (cur.c0 + CH > cur.n) {   // warp-uniform: slots past the set
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        const int p = cur.c0 + ((16 * mt + rot) & (CH - 1)) + g;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          if (p >= cur.n) s[nt][mt][0] = s[nt][mt][1] = -INFINITY;
          if (p + 8 >= cur.n) s[nt][mt][2] = s[nt][mt][3] = -INFINITY;
        }
      }
    }
    const bool last = !MULTI || cur.c0 + CH >= cur.n;   // the item's last unit
    if (last && nxt.bh >= 0) load_q(nxt);
    // ---- softmax over the rows of each column (columns 2t and 2t + 1 in this thread)
    constexpr int NP = PF == kProbMma3 ? 3 : PF == kProbCols4 ? 2 : 1;   // MMAs of a step
    uint32_t pr[NP][NT][MT][2];
    const uint32_t part_mask = t == 0 ? 0xFFFFFFFFu : t == 1 ? 0xFFFFu : 0u;   // kProbCols1
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      float x0 = -INFINITY, x1 = -INFINITY;
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        x0 = fmaxf(x0, fmaxf(s[nt][mt][0], s[nt][mt][2]));
        if (PF != kProbCols1) x1 = fmaxf(x1, fmaxf(s[nt][mt][1], s[nt][mt][3]));
      }
#pragma unroll
      for (int w = 4; w < 32; w <<= 1) {
        x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, w));
        if (PF != kProbCols1) x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, w));
      }
      if (PF == kProbCols1) x1 = x0;
      x0 *= sl2;
      x1 *= sl2;
      if (MULTI) {
        x0 = fmaxf(x0, m[nt][0]);
        x1 = fmaxf(x1, m[nt][1]);
        if (cur.c0 > 0) {
          const float f0 = ex2_fast(m[nt][0] - x0), f1 = ex2_fast(m[nt][1] - x1);
#pragma unroll
          for (int i = 0; i < DT; ++i) {
            o[nt][i][0] *= f0;
            o[nt][i][1] *= f1;
            o[nt][i][2] *= f0;
            o[nt][i][3] *= f1;
          }
          l[nt][0] *= f0;
          l[nt][1] *= f1;
        }
        m[nt][0] = x0;
        m[nt][1] = x1;
      }
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int half = 0; half < 2; ++half) {   // rows g and g + 8
          const float p0 = ex2_fast(fmaf(s[nt][mt][2 * half], sl2, -x0));
          if (PF == kProbCols1) {   // every column is the head: hi, mid and lo in columns 0, 1 and 2
            const float r = below_bf16(p0), lo = below_bf16(r);
            pr[0][nt][mt][half] = movm_t(upper_halves(t == 0 ? p0 : lo, r) & part_mask);
            continue;
          }
          const float p1 = ex2_fast(fmaf(s[nt][mt][2 * half + 1], sl2, -x1));
          if (PF == kProbBf16) {
            pr[0][nt][mt][half] = movm_t(pack_bf16(p0, p1));
            continue;
          }
          if (NP > 1) {   // this lane's rows of the columns' sums
            l[nt][0] += p0;
            l[nt][1] += p1;
          }
          const float r0 = below_bf16(p0), r1 = below_bf16(p1);
          const uint32_t hi = upper_halves(p0, p1), mid = upper_halves(r0, r1);
          const uint32_t lo = upper_halves(below_bf16(r0), below_bf16(r1));
          if (PF == kProbCols2) {   // columns 2t, 2t + 1: part t of the heads (part 3: zero)
            pr[0][nt][mt][half] = movm_t(t == 0 ? hi : t == 1 ? mid : t == 2 ? lo : 0u);
          } else if (PF == kProbCols4) {   // columns 4..7: the heads' middle parts
            pr[0][nt][mt][half] = movm_t(t < 2 ? hi : mid);
            pr[NP - 1][nt][mt][half] = movm_t(t < 2 ? lo : 0u);
          } else {
            pr[0][nt][mt][half] = movm_t(hi);
            pr[NP / 2][nt][mt][half] = movm_t(mid);
            pr[NP - 1][nt][mt][half] = movm_t(lo);
          }
        }
    }
    // acc += rows^T P^T of step mt; the smaller parts are summed first, so that a step rounds the
    // accumulator twice at most
    auto add_parts = [&](float (&acc)[4], uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3, int nt, int mt) {
      if (NP > 1) {
        float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int n = NP - 1; n > 0; --n) mma_bf16(e, x0, x1, x2, x3, pr[n][nt][mt][0], pr[n][nt][mt][1]);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += e[k];
      }
      mma_bf16(acc, x0, x1, x2, x3, pr[0][nt][mt][0], pr[0][nt][mt][1]);
    };
    // ---- O^T += V_rows^T P^T, and, of single MMAs, the row sums from a row of ones
#pragma unroll
    for (int ti = 0; ti < TPC; ++ti) {
      cp_async_wait_group<kRgStages - 1>();
      __syncwarp();
#pragma unroll
      for (int mk = 0; mk < MPT; ++mk) {
        const int mt = ti * MPT + mk;
#pragma unroll
        for (int i = 0; i < DT; ++i) {   // dims 16 i .. 16 i + 15
          uint32_t x[4];
          ldsm4_t(va[i & 3] + ((TPC + ti) % kRgStages) * kRgTile + mk * 16 * C::kRow +
                      (i >> 2) * 128,
                  x);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
            add_parts(o[nt][i], x[0], x[1], x[2], x[3], nt, mt);
        }
        constexpr uint32_t kOnes = 0x3F803F80u;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
          if (NP == 1) mma_bf16(l[nt], kOnes, kOnes, kOnes, kOnes, pr[0][nt][mt][0], pr[0][nt][mt][1]);
      }
      copy_ahead(TPC + ti);
    }
    // ---- normalised rows out: transposed through the query buffer, whole rows stored
    if (last) {
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        // the parts of a head in other columns
        auto join = [](float& a, float& b) {   // columns 2t and 2t + 1 of a row
          if (PF == kProbCols1) {   // 0, 1, 2 and 3
            a += b;
            a += __shfl_xor_sync(0xffffffffu, a, 1);
          } else if (PF == kProbCols2) {   // 2t and 2t + 1, for every t
            a += __shfl_xor_sync(0xffffffffu, a, 1);
            b += __shfl_xor_sync(0xffffffffu, b, 1);
          }
          if (PF == kProbCols2 || PF == kProbCols4) {   // c and c + 4
            a += __shfl_xor_sync(0xffffffffu, a, 2);
            b += __shfl_xor_sync(0xffffffffu, b, 2);
          }
        };
#pragma unroll
        for (int i = 0; i < DT; ++i) {
          join(o[nt][i][0], o[nt][i][1]);
          join(o[nt][i][2], o[nt][i][3]);
        }
        if (NP == 1) {
          join(l[nt][0], l[nt][1]);
        } else {
#pragma unroll
          for (int w = 4; w < 32; w <<= 1) {
            l[nt][0] += __shfl_xor_sync(0xffffffffu, l[nt][0], w);
            l[nt][1] += __shfl_xor_sync(0xffffffffu, l[nt][1], w);
          }
        }
        const float i0 = 1.f / l[nt][0], i1 = 1.f / l[nt][1];
#pragma unroll
        for (int i2 = 0; i2 < DT / 2; ++i2) {   // chunks 4 i2 .. 4 i2 + 3 (8 dims each)
          uint32_t w[4];
#pragma unroll
          for (int k = 0; k < 4; ++k)
            w[k] = pack_bf16(o[nt][2 * i2 + (k >> 1)][2 * (k & 1)] * i0,
                             o[nt][2 * i2 + (k >> 1)][2 * (k & 1) + 1] * i1);
          stsm4_t(qa[i2 & 1] + nt * 8 * C::kRow + (i2 >> 1) * 128, w[0], w[1], w[2], w[3]);
        }
      }
      __syncwarp();
      uint32_t odd = 0u;   // NaN where a value is not finite
#pragma unroll
      for (int i = 0; i < QV; ++i) {
        const int e = i * 32 + lane, h = e / C::kLpr, c = e % C::kLpr;
        if (h < G) {
          const uint4 w = ld_shared_v4(qbuf + h * C::kRow + ((((c & 7) ^ (h & 7)) | (c & ~7)) << 4));
          *reinterpret_cast<uint4*>(static_cast<uint16_t*>(a.out) +
                                    ((int64_t(cur.bh) * G + h) * d.N + cur.u) * D + 8 * c) = w;
          odd = zero_times(w.w, zero_times(w.z, zero_times(w.y, zero_times(w.x, odd))));
        }
      }
      if (__any_sync(0xffffffffu, odd != 0u)) {
        __syncwarp();
        redo_non_finite<D>(a, cur.bh, cur.u, FULL ? cur.u + 1 : cur.n, FULL ? nullptr : sel_c - cur.c0 - 8 * grp);
      }
    }
    cur = nxt;
    sel_c = sel_n;
    if (cur.bh >= 0) nxt = next_unit(cur);
    next_sel();
    if (2 * TPC == kRgStages) load_idx(nxt, sel_n, 0);   // the unit after next was not known before
  }
  cp_async_wait_group<0>();
}

template <int D, int NT, int PF, int CH, bool MULTI, bool FULL>
cudaError_t launch_gather(const ReplayArgs& a, int num_sms, cudaStream_t st) {
  using C = Rg<D, NT>;
  static_assert(C::kSmem <= 232448 - 32, "shared memory budget");
  auto kernel = replay_gather_kernel<D, NT, PF, CH, MULTI, FULL>;
  static SmemOptIn smem;
  if (cudaError_t e = smem(kernel, C::kSmem)) return e;
  const int64_t items = int64_t(a.d.B) * a.d.Hkv * a.d.N;
  const int grid = static_cast<int>(items < num_sms ? items : num_sms);   // persistent
  return launch_kernel(a.overlap, kernel, grid, 32 * C::kWarps, C::kSmem, st, a);
}

// Sets of one unit (guided, S <= 128).
template <int D, int NT, int PF>
cudaError_t launch_gather_one(const ReplayArgs& a, int num_sms, cudaStream_t st) {
  const int unit = replay_gather_unit(a.d);
  if constexpr (D == 128)
    if (unit == 32) return launch_gather<D, NT, PF, 32, false, false>(a, num_sms, st);
  return unit == 64 ? launch_gather<D, NT, PF, 64, false, false>(a, num_sms, st)
                    : launch_gather<D, NT, PF, 128, false, false>(a, num_sms, st);
}

// Sets of any size, 64 rows at a time.
template <int D, int NT, int PF>
cudaError_t launch_gather_multi(const ReplayArgs& a, int num_sms, cudaStream_t st) {
  return a.full ? launch_gather<D, NT, PF, 64, true, true>(a, num_sms, st)
                : launch_gather<D, NT, PF, 64, true, false>(a, num_sms, st);
}

template <int D>
cudaError_t launch_gather_d(const ReplayArgs& a, int num_sms, cudaStream_t st) {
  const int G = a.d.Hq / a.d.Hkv;
  if (a.full || a.d.S > 128)
    return G == 1   ? launch_gather_multi<D, 1, kProbCols1>(a, num_sms, st)
           : G == 2 ? launch_gather_multi<D, 1, kProbCols2>(a, num_sms, st)
           : G <= 4 ? launch_gather_multi<D, 1, kProbCols4>(a, num_sms, st)
           : G <= 8 ? launch_gather_multi<D, 1, kProbMma3>(a, num_sms, st)
                    : launch_gather_multi<D, 2, kProbMma3>(a, num_sms, st);
  // d = 128 sets of at most 128 rows take bf16 probabilities, like the full-attention
  // kernel; everything else keeps fp32 probabilities in three parts
  if constexpr (D == 128)
    return G <= 8 ? launch_gather_one<D, 1, kProbBf16>(a, num_sms, st)
                  : launch_gather_one<D, 2, kProbBf16>(a, num_sms, st);
  else
    return G == 1   ? launch_gather_one<D, 1, kProbCols1>(a, num_sms, st)
           : G == 2 ? launch_gather_one<D, 1, kProbCols2>(a, num_sms, st)
           : G <= 4 ? launch_gather_one<D, 1, kProbCols4>(a, num_sms, st)
           : G <= 8 ? launch_gather_one<D, 1, kProbMma3>(a, num_sms, st)
                    : launch_gather_one<D, 2, kProbMma3>(a, num_sms, st);
}

}  // namespace

// Rows per unit: the smallest of 32, 64 and 128 that holds a set of S rows (32 only where a
// unit then still has the two key tiles that the tile stream needs, d = 128); sets past 128
// rows go 64 at a time, whose score registers leave room for the running output.
int replay_gather_unit(const ReplayDims& d) {
  if (d.S > 128) return 64;
  if (d.S <= 32 && d.d == 128) return 32;
  return d.S <= 64 ? 64 : 128;
}

cudaError_t launch_replay_gather(const ReplayArgs& a, int num_sms, cudaStream_t st) {
  return a.d.d == 128 ? launch_gather_d<128>(a, num_sms, st)
                      : launch_gather_d<64>(a, num_sms, st);
}

}  // namespace mot
