// Tiles of the kernels that read raw frames themselves (lpa_mean, lpa_grad): 64 pixels wide, the raw
// footprint of every sensor fetched in groups of eight samples and converted into shared memory.
#pragma once
#include "lpa_convert.cuh"
#include "lpa_launch.h"

namespace lpa {

constexpr int kBW = LPA_MEAN_TILE_W;

// First candidate cell of a window along one axis of one colour phase: the position is cell `l` (from
// the box origin, even) plus fraction f; the window reaches h (m = floor(h / 2)). Returns the
// lattice index (cell o + 2 i) and its offset from the position.
__device__ __forceinline__ int first_cell(int l, float f, int o, float h, float m, float &delta) {
  const int e = l - o;
  const float r = (e & 1) ? f + 1.f : f;             // position from the even lattice cell below, in [0, 2)
  const float n = (h - r) * 0.5f < m ? m - 1.f : m;  // floor((h - r) / 2)
  delta = -2.f * n - r;
  return (e >> 1) - (int)n;
}

// A first cell as it is where the window's cells lie in the box, else (negative ones included) the last
// that does: one unsigned minimum; the caller compares to record the move.
__device__ __forceinline__ int cell_in(int i, int last) { return (int)min((unsigned)i, (unsigned)last); }

// A group of eight columns of one row of a sensor's box: where it lies and its raw samples, zeros off the frame.
struct Group {
  int s, row, col, X, Y;
  uint4 q;
};

// Box origin of a tile in sensor s: x on a multiple of 8 (16-byte loads), y even. FP32 is enough
// (the box has a margin of a pixel). The fetch and the position tables form it each for themselves and must get the
// same integers, so every rounding is written out: a sum that the compiler fused in one place and not in
// another could fall on two sides of an integer.
__device__ __forceinline__ int2 box_origin(const LpaSensorK &S, int u0, int v0, int bh) {
  auto origin = [&](float gu, float gv, float gt, float ext) {
    const float u = (float)(gu < 0.f ? u0 + kBW - 1 : u0), v = (float)(gv < 0.f ? v0 + bh - 1 : v0);
    const float q = __fsub_rn(__fadd_rn(__fmaf_rn(gv, v, __fmul_rn(gu, u)), gt), ext);
    return (int)floorf(fminf(fmaxf(q, -LPA_FAR_F), LPA_FAR_F));
  };
  return make_int2(origin(S.Gf[0], S.Gf[1], S.Gt[0], S.ext_x) & ~7, origin(S.Gf[2], S.Gf[3], S.Gt[1], S.ext_y) & ~1);
}

__device__ __forceinline__ Group load_group(const LpaLaunch &L, int s, int g, int u0, int v0, int bh) {
  const LpaSensorK &S = L.s[s];
  const int2 o = box_origin(S, u0, v0, bh);
  Group r;
  r.s = s;
  r.row = (int)__umulhi((unsigned)g, S.group_magic);
  r.col = g - r.row * (S.box_w >> 3);
  r.X = o.x + 8 * r.col;
  r.Y = o.y + r.row;
  r.q = make_uint4(0, 0, 0, 0);
  if (r.X >= 0 && r.X < S.width && r.Y >= 0 && r.Y < S.height)
    r.q = __ldg(reinterpret_cast<const uint4 *>(S.raw + (size_t)r.Y * S.raw_pitch + r.X));
  return r;
}

// Fetch the boxes of sensors s0 .. s1 - 1, two 16-byte loads in flight per thread of NT, and hand each group
// to put(group).
template <int NT, class Put>
__device__ __forceinline__ void stage_boxes(const LpaLaunch &L, int s0, int s1, int u0, int v0, int bh, Put &&put) {
  int total = 0;
  for (int s = s0; s < s1; s++) total += (L.s[s].box_w >> 3) * L.s[s].box_h;
  auto fetch = [&](int k) {
    int s = s0, n = (L.s[s0].box_w >> 3) * L.s[s0].box_h;
    while (k >= n) k -= n, s++, n = (L.s[s].box_w >> 3) * L.s[s].box_h;
    return load_group(L, s, k, u0, v0, bh);
  };
  for (int k = threadIdx.x; k < total; k += 2 * NT) {
    const bool two = k + NT < total;
    const Group a = fetch(k);
    if (two) {
      const Group b = fetch(k + NT);
      put(a);
      put(b);
    } else {
      put(a);
    }
  }
}

}  // namespace lpa
