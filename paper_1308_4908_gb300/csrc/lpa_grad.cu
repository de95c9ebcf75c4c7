// Pass 1 of the adaptive reconstruction (Section 5.4): the gradient of the order-1 fit of the green channel
// at one scale, for windows of at most 4 x 4 cells of a colour phase.
//
// The general kernel in its gradient mode searches six windows of about five samples per pixel of a
// three-sensor rig and stages all four colour phases, of which the pass reads two, behind a conversion
// pass of the whole frame: 170 us for 1920 x 1080 (issue 75 %, a fifth of the FP64 pipe for the per-tile
// positions of 16 x 16 pixels). Here, as in lpa_mean, the candidate cells are a fixed N x N block from
// the window's first cell, the raw footprints of 64 x 8 P pixels are fetched and only green samples
// converted, and each thread takes P pixels one after the other. Warps hold every second pixel of a row
// at 1x (the phase class of the output scale, as PixelMap), so that a cell outside the window is
// skipped by the whole warp. Positions, offsets, window values and sums are formed by the general
// kernel's operations in its order: the gradients are the same bits, so the steering matrices and the interval
// rule that follow are too. 1920 x 1080, three sensors: 170 us with the conversion pass before, 116 us.
#include "lpa_dispatch.h"
#include "lpa_kernel.cuh"
#include "lpa_tile.cuh"

namespace lpa {
namespace {

constexpr int kThreads = 512;

// Column of a 64-pixel row taken by position t: pixels equal modulo sx one class after the other.
__device__ __forceinline__ int class_column(int t, int sx) {
  switch (sx) {
    case 2: return 2 * (t & 31) + (t >> 5);
    case 3: return t < 22 ? 3 * t : t < 43 ? 3 * (t - 22) + 1 : 3 * (t - 43) + 2;
    case 4: return 4 * (t & 15) + (t >> 4);
    default: return t;
  }
}

// The green samples of a group into the sensor's two planes (phase (1, 0): even rows, odd columns; phase
// (0, 1): odd rows, even columns).
__device__ __forceinline__ void store_green(const LpaLaunch &L, const Group &r, float2 *planes) {
  const LpaSensorK &S = L.s[r.s];
  const int PW = S.box_w >> 1, PP = PW * (S.box_h >> 1);
  const int n = r.X >= 0 && r.Y >= 0 && r.Y < S.height ? S.width - r.X : 0;  // columns inside the frame
  const int odd = (r.row & 1) ? 0 : 1;  // the green columns of this row
  const uint32_t w[4] = {r.q.x, r.q.y, r.q.z, r.q.w};
  float2 v[4];  // (f, 1 / s2)
  float y[4];
#pragma unroll
  for (int k = 0; k < 4; k++) y[k] = (float)(odd ? w[k] >> 16 : w[k] & 0xffffu);
  if (S.plain) {
#pragma unroll
    for (int k = 0; k < 4; k += 2) {
      float2 f, iv;
      convert_two(S, y[k], y[k + 1], 2 * k + odd < n, 2 * k + 2 + odd < n, f, iv);
      v[k] = make_float2(f.x, iv.x);
      v[k + 1] = make_float2(f.y, iv.y);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; k++)
      v[k] = 2 * k + odd < n ? convert_sample<false>(S, false, r.X + 2 * k + odd, r.Y, y[k]) : make_float2(0.f, 0.f);
  }
  float4 *o = reinterpret_cast<float4 *>(planes + (r.row & 1) * PP + (r.row >> 1) * PW + 4 * r.col);
  o[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  o[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
}

template <int N, bool F64, int P>
__global__ void __launch_bounds__(kThreads, 2) lpa_grad(const __grid_constant__ LpaLaunch L) {
  constexpr int BH = 8 * P;
  if (*reinterpret_cast<volatile unsigned int *>(L.status) & LPA_ERR_TIMEOUT) return;
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x, S = L.n_sensors;
  const int u0 = (int)blockIdx.x * kBW, v0 = (int)blockIdx.y * BH;
  // positions of the tile's 8 x 8 blocks, relative to each box's origin
  int4 *anchor = reinterpret_cast<int4 *>(smem + L.mean_tab);
  for (int k = tid; k < S * BH; k += kThreads) {
    const int s = k / BH, b = k - s * BH;
    const LpaSensorK &Sk = L.s[s];
    const int2 o = box_origin(Sk, u0, v0, BH);
    const double uu = u0 + 8 * (b & 7), vv = v0 + 8 * (b >> 3);
    const double qx = fmin(fmax(Sk.G[0] * uu + Sk.G[1] * vv + Sk.G[2], -LPA_FAR), LPA_FAR);
    const double qy = fmin(fmax(Sk.G[3] * uu + Sk.G[4] * vv + Sk.G[5], -LPA_FAR), LPA_FAR);
    const double fx = floor(qx), fy = floor(qy);
    anchor[k] = make_int4((int)fx - o.x, (int)fy - o.y, __float_as_int((float)(qx - fx)), __float_as_int((float)(qy - fy)));
  }
  stage_boxes<kThreads>(L, 0, S, u0, v0, BH,
                        [&](const Group &r) { store_green(L, r, reinterpret_cast<float2 *>(smem + r.s * L.mean_plane)); });
  __syncthreads();

  const int col = class_column(tid & 63, (L.px_map & 3) + 1), u = u0 + col;
  const float log2e = 1.4426950408889634f;
  const float sg = L.sigma[0] * L.green_ratio;
  const float R = L.trunc_k * sg, R2 = R * R, cexp = -log2e / (2.f * sg * sg);
#pragma unroll 1
  for (int k = 0; k < P; k++) {
    const int row = (tid >> 6) * P + k, v = v0 + row;
    MomentsLean<1> m;
    m.zero();
    int moved = 0;
#pragma unroll 1
    for (int s = 0; s < S; s++) {
      const LpaSensorK &Sk = L.s[s];
      const int4 an = anchor[s * BH + (row >> 3) * 8 + (col >> 3)];
      const float du = (float)(col & 7), dv = (float)(row & 7);
      const float px = fmaf(dv, Sk.Gf[1], fmaf(du, Sk.Gf[0], __int_as_float(an.z)));
      const float py = fmaf(dv, Sk.Gf[3], fmaf(du, Sk.Gf[2], __int_as_float(an.w)));
      const float flx = floorf(px), fly = floorf(py);
      const int lx = an.x + (int)flx, ly = an.y + (int)fly;
      const float fx = px - flx, fy = py - fly;
      const float hx = R * Sk.hx_unit + 1e-3f, hy = R * Sk.hy_unit + 1e-3f;
      const float mx = floorf(0.5f * hx), my = floorf(0.5f * hy);
      const float a00 = Sk.A[0], a01 = Sk.A[1], a10 = Sk.A[2], a11 = Sk.A[3];
      const float2 T2 = make_float2(2.f * a01, 2.f * a11), S2 = make_float2(2.f * a00, 2.f * a10);
      const int PW = Sk.box_w >> 1, PH = Sk.box_h >> 1;
#pragma unroll
      for (int sub = 0; sub < 2; sub++) {
        const int ox = 1 - sub, oy = sub;
        float Dx0, Dy0;
        const int i0 = first_cell(lx, fx, ox, hx, mx, Dx0), j0 = first_cell(ly, fy, oy, hy, my, Dy0);
        const int i = cell_in(i0, PW - N), j = cell_in(j0, PH - N);
        moved |= (i ^ i0) | (j ^ j0);
        const float2 *pl = reinterpret_cast<const float2 *>(smem + s * L.mean_plane) + sub * (PW * PH) + j * PW + i;
        const float2 DR0 = make_float2(fmaf(a00, Dx0, a01 * Dy0), fmaf(a10, Dx0, a11 * Dy0));
#pragma unroll
        for (int r = 0; r < N; r++) {
          float2 D = __ffma2_rn(make_float2((float)r, (float)r), T2, DR0);
#pragma unroll
          for (int c = 0; c < N; c++, D = __fadd2_rn(D, S2))
            window_cell<1, LPA_GRADIENTS>(m, D, pl[r * PW + c], R2, cexp, L.taper, make_float4(1.f, 0.f, 1.f, 0.f));
        }
      }
      if (moved && u < L.out_w && v < L.out_h && abs(lx) < (1 << 20) && abs(ly) < (1 << 20)) atomicOr(L.status, LPA_ERR_BOUNDS);
    }
    const FitOut f = solve_with_fallback<3, MomentsLean<1>, true, F64>(m, L.min_pivot, L.cond_fallback);
    if (u < L.out_w && v < L.out_h) {
      float *g = L.aux + ((size_t)v * L.out_w + u) * 2;
      g[0] = f.valid ? f.c1 : 0.f;
      g[1] = f.valid ? f.c2 : 0.f;
    }
  }
}

template <int N, int P>
const void *pick(bool f64) {
  return f64 ? (const void *)lpa_grad<N, true, P> : (const void *)lpa_grad<N, false, P>;
}

}  // namespace
}  // namespace lpa

cudaError_t lpa_launch_grad(const LpaLaunch &L, bool f64, cudaStream_t st) {
  const void *fn = L.mean_size == 2 ? (L.mean_p == 1 ? lpa::pick<3, 1>(f64) : lpa::pick<3, 2>(f64))
                                    : (L.mean_p == 1 ? lpa::pick<4, 1>(f64) : lpa::pick<4, 2>(f64));
  cudaError_t e = lpa_opt_in(fn);
  if (e != cudaSuccess) return e;
  const int bh = lpa_mean_tile_h(L.mean_p);
  const dim3 grid((unsigned)((L.out_w + LPA_MEAN_TILE_W - 1) / LPA_MEAN_TILE_W), (unsigned)((L.out_h + bh - 1) / bh));
  void *args[] = {const_cast<LpaLaunch *>(&L)};
  return cudaLaunchKernel(fn, grid, dim3(lpa::kThreads), args, L.smem_bytes, st);
}
