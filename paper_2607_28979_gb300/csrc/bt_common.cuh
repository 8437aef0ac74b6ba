// Device helpers shared by the backbone-translator kernels: bt.cu (the stages one by one)
// and bt_scan.cu (the whole scan of a tile).
#pragma once

#include <cuda_bf16.h>

#include "bt_internal.h"
#include "ptx.cuh"

namespace mot {
namespace {

constexpr float kLnEps = 1e-5f;

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ int seq_len_of(const BtArgs& a, int b) {
  if (b >= a.batch) return 0;
  const int L = a.seq_lens[b];
  return L < 0 ? 0 : (L > a.d.S ? a.d.S : L);
}

struct GemmCfg {
  int mode;
  int K;          // reduction length per backbone
  int NT;         // accumulator columns per tile (multiple of 32, <= 256)
  int n_tiles;    // N tiles per group
  int groups;     // groups iterated (2E, or 2 for kBtOut)
  int row_tiles;  // row tiles per group
  int a_box_bytes;
  int b_rows_per_g;   // rows of the weight map per (group, slot) block
  int slots;          // kBtOut: window slots from a.slot on in this launch (else 0 or 1)
};

// One work item of the persistent loop. Every role decodes items the same way
// (skipping the same inactive tiles), so their barrier phases stay in step.
struct Work {
  int g, b, s0, ntok, j;
  int tok0;       // kBtOut: first token of the 128-token tile (routed: bucket position)
  int r;          // kBtOut: slot of the item, counted from a.slot
  int64_t row0;   // the tile's first row in its group's row space
  bool active;
};

// Items of a launch: dense, groups x row tiles x N tiles; routed, the tiles of
// every bucket (from the route kernel's prefix sums) x N tiles.
__device__ __forceinline__ int slot_items(const BtArgs& a, const GemmCfg& c) {
  if (!a.routed) return c.groups * c.row_tiles * c.n_tiles;
  const int* pre = a.rpre + (c.mode == kBtOut ? a.d.G + 1 : 0);
  return pre[a.d.G] * c.n_tiles;
}

__device__ __forceinline__ int total_items(const BtArgs& a, const GemmCfg& c) {
  return slot_items(a, c) * (c.slots > 1 ? c.slots : 1);
}

__device__ __forceinline__ Work decode(const BtArgs& a, const GemmCfg& c, int item) {
  Work w;
  w.r = 0;
  if (c.slots > 1) {
    const int per = slot_items(a, c);
    w.r = item / per;
    item -= w.r * per;
  }
  if (a.routed) {   // tile of bucket positions of group g
    const bool out = c.mode == kBtOut;
    const int* pre = a.rpre + (out ? a.d.G + 1 : 0);
    const int tile = item / c.n_tiles;
    w.j = item - tile * c.n_tiles;
    int g = 0;
    while (g + 1 < a.d.G && pre[g + 1] <= tile) ++g;
    w.g = g;
    const int span = out ? 128 : a.d.tau;
    const int pos0 = (tile - pre[g]) * span;
    w.ntok = min(span, a.cnt[g] - pos0);
    w.tok0 = pos0;
    w.b = 0;
    w.s0 = pos0;
    w.row0 = int64_t(pos0) * a.d.P;
    w.active = w.ntok > 0;
    return w;
  }
  const int per_g = c.row_tiles * c.n_tiles;
  w.g = item / per_g;
  const int rem = item - w.g * per_g;
  const int rt = rem / c.n_tiles;
  w.j = rem - rt * c.n_tiles;
  if (c.mode == kBtOut) {
    w.tok0 = rt * 128;
    w.b = w.tok0 / a.d.S;
    w.s0 = w.tok0 - w.b * a.d.S;
    w.ntok = 128;
    // active if any token of the tile is inside its sequence
    bool act = false;
    for (int b = w.b; b < a.d.B && b * a.d.S < w.tok0 + 128; ++b) {
      const int lo = max(0, w.tok0 - b * a.d.S);
      act = act || lo < seq_len_of(a, b);
    }
    w.active = act;
  } else {
    w.b = rt / a.d.tiles_b;
    w.s0 = (rt - w.b * a.d.tiles_b) * a.d.tau;
    w.ntok = min(a.d.tau, a.d.S - w.s0);
    w.tok0 = w.b * a.d.S + w.s0;
    w.active = w.s0 < seq_len_of(a, w.b);
  }
  w.row0 = int64_t(w.tok0) * a.d.P;
  return w;
}

// Whether token t of a (non-output) tile is a real token.
__device__ __forceinline__ bool tile_token_valid(const BtArgs& a, const Work& w, int t) {
  return t < w.ntok && (a.routed || w.s0 + t < seq_len_of(a, w.b));
}

// Named barrier over the nthreads epilogue threads, with the AND of p.
__device__ __forceinline__ bool epi_and(int id, int nthreads, bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred a, q;\n\t"
      "setp.ne.u32 a, %1, 0;\n\t"
      "bar.red.and.pred q, %2, %3, a;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(static_cast<uint32_t>(p)), "r"(id), "r"(nthreads)
      : "memory");
  return r != 0;
}

}  // namespace
}  // namespace mot
