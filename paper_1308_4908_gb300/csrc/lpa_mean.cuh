// Order 0 with one window scale: the local constant fit of Eq. 7, sum K f / s2 over sum K / s2.
//
// With one sum and one weight per sample the general kernel spends its instructions on finding the
// window (its bounding box, warp-wide maxima, rows, a test per cell): 2420 warp instructions per 32
// pixels of a two-sensor frame enlarged twofold, 300 per walk of a 9-cell window. Here the candidate
// cells of a window are a fixed N x N block of its colour phase (N = cells that a row or column of
// the window can hold), so the loops unroll, and a cell outside the window needs no test: its value
// exp(-r^2 / 2 sigma^2) - exp(-k^2 / 2) (Eq. 8) is not positive there and is cut at 0.
//
// A CTA of 512 threads reconstructs 64 x 8 P pixels, P rows per thread (kPeriodic on large frames: 256
// threads, P = 8, so that each cell and factor serves twice the rows: 187 -> 152 us enlarging 2 x 2048^2 twofold,
// 100 -> 93 us on the camera frame; three CTAs per SM, at two 173 and 96 us, at four 160 and 98 us); lanes are consecutive
// pixels of a row, so stores coalesce and neighbours read the same cells. The raw footprints of all sensors
// (of as many as two CTAs' shared memory holds) are read straight from global memory (16-byte loads,
// two in flight per thread) and converted once per sample (Eqs. 18 and 20) into colour-phase planes of
// (1 / s2, f / s2) in shared memory; one barrier later the sums of every sensor follow. Each cell is
// then one shared load and one paired FMA into (sum K / s2, sum K f / s2). No conversion pass goes
// ahead of the kernel: with 64 x 32 tiles (boxes of 80 x 42 samples at 1x) a sample is converted 1.64 times, and the
// pass cost 47 us of 517 on four 2336 x 1752 sensors. Measured against the general kernel with that pass: 2 x 2048^2 ->
// 4096^2 FP16 1226 -> 136 us, the four sensors (tabulated windows) 517 -> 84 us, 64^2 14.4 -> 6.3 us a call (2.9
// of it in the binding); 1024 x 900, three rotated sensors 147 -> 58 us, compensated 201 -> 106 us.
//
// kAxis: every sensor's axes are parallel to the output's, so the Gaussian factors into a column and
// a row factor, tabulated per tile: a cell is one FMA, one maximum, the load and the paired FMA.
// kPeriodic: besides, 2 or 4 output pixels span exactly one cell of a colour phase (translated sensors at
// 1x or twofold output), so pixels that far apart see the same offsets: a thread takes P rows of one
// class, forms the K of its cells once per sensor and slides the window down one cell a row, each
// loaded cell serving up to N rows. kFactored: the output is rotated against a sensor whose map is a
// rotation and an even scale, so |d|^2 still separates in the sensor's axes; the 2 N factors of a window are
// formed per pixel. kGeneral: each cell forms its offset and one exponential. kTabulated: kPeriodic at 1x on
// exactly translated sensors, whose window weights the caller may have tabulated (tab_weights): formed by the
// host in FP64 and rounded once, they are copied into shared memory instead of the factors.
#pragma once
#include <cuda_fp16.h>

#include <type_traits>

#include "lpa_launch.h"
#include "lpa_ptx.cuh"
#include "lpa_sums.cuh"
#include "lpa_tile.cuh"

namespace lpa {
namespace {

template <int NR, int NG>
struct Layout {
  static constexpr int kE = 2 * (NR + NG);       // factors: RB phase 0, RB phase 1, G phase 0, G phase 1
  static constexpr int kWords = 4 + kE;          // four first cells, then the factors
  static constexpr int kRow = (kWords + 3) / 4 * 4;
  // tabulated positions: words of a phase's weights (16-byte loads), the first of phase ph = ox + 2 oy in
  // a class, of a class (columns of unequal parity read different banks) and of a sensor (LpaLaunch::mean_k)
  static constexpr int kR = (NR * NR + 3) / 4 * 4, kG = (NG * NG + 3) / 4 * 4;
  __host__ __device__ static constexpr int phase_words(int ph) { return ph == 0 ? 0 : kR + (ph - 1) * kG; }
  static constexpr int kClass = (2 * (kR + kG) + 31) / 32 * 32 == 2 * (kR + kG) ? 2 * (kR + kG) + 4 : 2 * (kR + kG);
  static constexpr int kTab = 16 + 4 * kClass;
  static_assert(kTab >= 4 * kRow, "the tables of two classes per axis fit in the same place");
};

__device__ __forceinline__ void store_group(const LpaLaunch &L, const Group &r, float2 *planes) {
  const LpaSensorK &S = L.s[r.s];
  const int PW = S.box_w >> 1, PP = PW * (S.box_h >> 1);
  const int n = r.X >= 0 && r.Y >= 0 && r.Y < S.height ? S.width - r.X : 0;  // columns inside the frame
  const uint32_t w[4] = {r.q.x, r.q.y, r.q.z, r.q.w};
  float4 *even = reinterpret_cast<float4 *>(planes + 2 * (r.row & 1) * PP + (r.row >> 1) * PW + 4 * r.col);
  float4 *odd = even + (PP >> 1);
  float2 v[8];  // (1 / s2, f / s2)
  if (S.plain) {
#pragma unroll
    for (int k = 0; k < 4; k++) {
      float2 f, iv;
      convert_two(S, (float)(w[k] & 0xffffu), (float)(w[k] >> 16), 2 * k < n, 2 * k + 1 < n, f, iv);
      const float2 ivf = __fmul2_rn(iv, f);
      v[2 * k] = make_float2(iv.x, ivf.x);
      v[2 * k + 1] = make_float2(iv.y, ivf.y);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t y = (k & 1) ? w[k >> 1] >> 16 : w[k >> 1] & 0xffffu;
      v[k] = make_float2(0.f, 0.f);
      if (k < n) {
        const float2 fv = convert_sample<false>(S, false, r.X + k, r.Y, (float)y);  // (f, 1 / s2)
        v[k] = make_float2(fv.y, fv.y * fv.x);
      }
    }
  }
  even[0] = make_float4(v[0].x, v[0].y, v[2].x, v[2].y);
  even[1] = make_float4(v[4].x, v[4].y, v[6].x, v[6].y);
  odd[0] = make_float4(v[1].x, v[1].y, v[3].x, v[3].y);
  odd[1] = make_float4(v[5].x, v[5].y, v[7].x, v[7].y);
}

// Sums of one pixel and channel: (sum K / s2, sum K f / s2), or with what their additions rounded away
// (compensated).
template <bool COMP>
struct Sums {
  float2 h = {0.f, 0.f};
  __device__ __forceinline__ void add(float K, float2 cell) { h = __ffma2_rn(make_float2(K, K), cell, h); }
  __device__ __forceinline__ float2 value() const { return h; }
};
template <>
struct Sums<true> {
  float2 h = {0.f, 0.f}, l = {0.f, 0.f};
  __device__ __forceinline__ void add(float K, float2 cell) { comp_sum2(h, l, __fmul2_rn(make_float2(K, K), cell)); }
  __device__ __forceinline__ float2 value() const { return __fadd2_rn(h, l); }
};

enum { kGeneral = 0, kAxis = 1, kFactored = 2, kPeriodic = 3, kTabulated = 4 };

// The cells and factors of one position along one axis for every (window, phase): words of Layout at
// t[0], t[stride], ... `last`: how many cells further the last position served by the entry lies. Returns
// false if a first cell had to be moved so that all of them lie in the box.
template <int NR, int NG>
__device__ __forceinline__ bool axis_entry(const LpaLaunch &L, const LpaSensorK &Sk, bool col, int l, float f, int last, float *t,
                                           int stride) {
  const float log2e = 1.4426950408889634f;
  const float a = col ? Sk.A[0] : Sk.A[3];
  const int cells = (col ? Sk.box_w : Sk.box_h) >> 1, step = col ? 1 : Sk.box_w >> 1;
  bool ok = true;
#pragma unroll
  for (int g = 0; g < 2; g++) {
    const int N = g ? NG : NR;
    const float sg = g ? L.sigma[0] * L.green_ratio : L.sigma[0];
    const float h = L.trunc_k * sg * (col ? Sk.hx_unit : Sk.hy_unit) + 1e-3f, m = floorf(0.5f * h);
    const float c = -log2e / (2.f * sg * sg) * a * a;
#pragma unroll
    for (int ph = 0; ph < 2; ph++) {
      float d;
      const int i = first_cell(l, f, ph, h, m, d), at = max(min(i, cells - N - last), 0);
      ok = ok && i == at;
      t[(2 * g + ph) * stride] = __int_as_float(at * step);
      float *w = t + (4 + 2 * NR * g + N * ph) * stride;
#pragma unroll
      for (int j = 0; j < N; j++) {
        const float dj = d + 2.f * (float)j;
        w[j * stride] = ex2_approx(c * dj * dj);
      }
    }
  }
  return ok;
}

template <int NR, int NG, int FORM, int P, bool COMP>
__global__ void __launch_bounds__(lpa_mean_threads(P), P == 8 ? 3 : 2) lpa_mean(const __grid_constant__ LpaLaunch L) {
  using T = Layout<NR, NG>;
  constexpr int kThreads = lpa_mean_threads(P), BH = lpa_mean_tile_h(P);
  // read now, looked at before the stores: once a bounded wait has run out, nothing is written
  const unsigned int status = *reinterpret_cast<volatile unsigned int *>(L.status);
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x, S = L.n_sensors;
  const int y_end = L.mean_y1;
  const int u0 = (int)blockIdx.x * kBW, v0 = L.mean_y0 + (int)blockIdx.y * BH;
  const float log2e = 1.4426950408889634f;
  const float sg[2] = {L.sigma[0], L.sigma[0] * L.green_ratio};

  // positions of the tile's columns and rows (AXIS) or of its 8 x 8 blocks' corners, in FP64
  float *xt = reinterpret_cast<float *>(smem + L.mean_tab);
  float *yt = xt + S * T::kWords * kBW;
  int4 *anchor = reinterpret_cast<int4 *>(smem + L.mean_tab);
  const int lx = L.mean_lx, ly = L.mean_ly, tx = 1 << lx, ty = 1 << ly;  // kPeriodic: pixels to a cell
  if constexpr (FORM == kTabulated) {
    for (int w = kThreads - 1 - tid; w < S * T::kTab; w += kThreads) {  // the last threads first: the others fetch samples
      const int s = w / T::kTab, r = w - s * T::kTab;
      float v = __ldg(L.mean_k + w);
      if (r < 16) {  // a first column or row, from the pixel's cell to the box
        const LpaSensorK &Sk = L.s[s];
        const int2 o = box_origin(Sk, u0, v0, BH);
        const bool col = r < 8;
        const int ph = (r >> 1) & 3, c = r & 1, N = ph == 1 || ph == 2 ? NG : NR;
        const int l = (col ? u0 + Sk.ix_shift - o.x - (ph & 1) : v0 + Sk.iy_shift - o.y - (ph >> 1)) + c;
        const int i = (l >> 1) + __float_as_int(v), last = col ? (kBW - 1) >> 1 : (BH - 1) >> 1;
        const int at = max(min(i, ((col ? Sk.box_w : Sk.box_h) >> 1) - N - last), 0);
        if (at != i && (col ? u0 + c < L.out_w : v0 + c < y_end)) atomicOr(L.status, LPA_ERR_BOUNDS);
        v = __int_as_float(col ? at : at * (Sk.box_w >> 1));
      }
      xt[w] = v;
    }
  } else if constexpr (FORM == kPeriodic) {
    // one entry per sensor, axis and class of positions: class c starts at G c + G_t, and the n-th
    // pixel of a class lies exactly 2 n px further, whatever the tile
    const int entry = kThreads - 1 - tid;  // by the last threads: the first ones fetch samples
    if (entry < S * (tx + ty)) {
      const int s = entry / (tx + ty), e = entry - s * (tx + ty);
      const bool col = e < tx;
      const int c = col ? e : e - tx;
      const LpaSensorK &Sk = L.s[s];
      const int2 o = box_origin(Sk, u0, v0, BH);
      const double q = fmin(fmax(col ? Sk.G[0] * c + Sk.G[2] : Sk.G[4] * c + Sk.G[5], -LPA_FAR), LPA_FAR), fl = floor(q);
      const int l = (int)fl + (col ? 2 * (u0 >> lx) - o.x : 2 * (v0 >> ly) - o.y);
      float *t = xt + entry * T::kRow;
      const int last = col ? (kBW - 1) >> lx : (BH - 1) >> ly;
      if (!axis_entry<NR, NG>(L, Sk, col, l, (float)(q - fl), last, t, 1) && (col ? u0 + c < L.out_w : v0 + c < y_end) && fabs(q) < 1e6)
        atomicOr(L.status, LPA_ERR_BOUNDS);
    }
  } else if constexpr (FORM == kAxis) {
    for (int k = tid; k < S * (kBW + BH); k += kThreads) {
      const int s = k / (kBW + BH), e = k - s * (kBW + BH);
      const bool col = e < kBW;
      const LpaSensorK &Sk = L.s[s];
      const int2 o = box_origin(Sk, u0, v0, BH);
      const double q = fmin(fmax(col ? Sk.G[0] * (u0 + e) + Sk.G[2] : Sk.G[4] * (v0 + e - kBW) + Sk.G[5], -LPA_FAR), LPA_FAR);
      const double fl = floor(q);
      const int l = (int)fl - (col ? o.x : o.y);
      float *t = col ? xt + s * T::kWords * kBW + e : yt + (s * BH + e - kBW) * T::kRow;
      if (!axis_entry<NR, NG>(L, Sk, col, l, (float)(q - fl), 0, t, col ? kBW : 1) &&
          (col ? u0 + e < L.out_w : v0 + e - kBW < y_end) && fabs(q) < 1e6)
        atomicOr(L.status, LPA_ERR_BOUNDS);
    }
  } else {
    constexpr int NA = BH;  // 8 x 8 blocks of the tile
    for (int k = tid; k < S * NA; k += kThreads) {
      const int s = k / NA, b = k - s * NA;
      const LpaSensorK &Sk = L.s[s];
      const int2 o = box_origin(Sk, u0, v0, BH);
      const double uu = u0 + 8 * (b & 7), vv = v0 + 8 * (b >> 3);
      const double qx = fmin(fmax(Sk.G[0] * uu + Sk.G[1] * vv + Sk.G[2], -LPA_FAR), LPA_FAR);
      const double qy = fmin(fmax(Sk.G[3] * uu + Sk.G[4] * vv + Sk.G[5], -LPA_FAR), LPA_FAR);
      const double fx = floor(qx), fy = floor(qy);
      anchor[k] = make_int4((int)fx - o.x, (int)fy - o.y, __float_as_int((float)(qx - fx)), __float_as_int((float)(qy - fy)));
    }
  }

  // this thread's column and its P rows: row0 + k, or (kPeriodic) row0 + ty k
  const int col = (tid & 31) + 32 * ((tid >> 5) & 1), group = tid >> 6;
  constexpr bool kClasses = FORM == kPeriodic || FORM == kTabulated;
  const int row0 = kClasses ? (group >> ly) * (P << ly) + (group & (ty - 1)) : group * P;
  const int u = u0 + col;
  Sums<COMP> acc[P][3];  // per row and channel

  // the sensors of one filling of the plane buffers at a time (all of them, unless they are many)
#pragma unroll 1
  for (int s0 = 0; s0 < S; s0 += L.mean_bufs) {
    const int s1 = min(S, s0 + L.mean_bufs);
    if (s0) __syncthreads();  // the buffers' readers have left them
    stage_boxes<kThreads>(L, s0, s1, u0, v0, BH, [&](const Group &r) {
      store_group(L, r, reinterpret_cast<float2 *>(smem + (r.s - s0) * L.mean_plane));
    });
    __syncthreads();  // the planes (and the position tables) are whole
#pragma unroll 1
  for (int s = s0; s < s1; s++) {
    const LpaSensorK &Sk = L.s[s];
    const float2 *planes = reinterpret_cast<const float2 *>(smem + (s - s0) * L.mean_plane);
    const int PW = Sk.box_w >> 1, PP = PW * (Sk.box_h >> 1);
    if constexpr (kClasses) {
      const float *ex = xt + (s * (tx + ty) + (col & (tx - 1))) * T::kRow;
      const float *ey = xt + (s * (tx + ty) + tx + (group & (ty - 1))) * T::kRow;
      const int shift = (col >> lx) + (group >> ly) * P * PW;  // whole cells from the class's first pixel
      auto phase = [&](auto N_, auto c_, int ox, int oy, int g) {
        constexpr int N = decltype(N_)::value, c = decltype(c_)::value;
        float K[N][N];
        const float2 *pl;
        if constexpr (FORM == kTabulated) {
          const int pu = col & 1, pv = group & 1, ph = ox + 2 * oy;
          const float *t = xt + s * T::kTab;
          const float4 *k = reinterpret_cast<const float4 *>(t + 16 + (2 * pv + pu) * T::kClass + T::phase_words(ph));
#pragma unroll
          for (int j = 0; j < N * N; j += 4) {
            const float4 q = k[j / 4];
            const float e[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int i = 0; i < 4; i++)
              if (j + i < N * N) K[(j + i) / N][(j + i) % N] = e[i];
          }
          pl = planes + ph * PP + shift + __float_as_int(t[2 * ph + pu]) + __float_as_int(t[8 + 2 * ph + pv]);
        } else {
          const float *fx = ex + 4 + 2 * NR * g + N * ox, *fy = ey + 4 + 2 * NR * g + N * oy;
#pragma unroll
          for (int j = 0; j < N; j++)
#pragma unroll
            for (int i = 0; i < N; i++) K[j][i] = fmaxf(fmaf(fx[i], fy[j], -L.taper), 0.f);
          pl = planes + (ox + 2 * oy) * PP + shift + __float_as_int(ex[2 * g + ox]) + __float_as_int(ey[2 * g + oy]);
        }
#pragma unroll
        for (int r = 0; r < N + P - 1; r++)
#pragma unroll
          for (int i = 0; i < N; i++) {
            const float2 cell = pl[r * PW + i];
#pragma unroll
            for (int k = 0; k < P; k++)
              if (r - k >= 0 && r - k < N) acc[k][c].add(K[r - k][i], cell);
          }
      };
      phase(std::integral_constant<int, NR>(), std::integral_constant<int, 0>(), 0, 0, 0);
      phase(std::integral_constant<int, NG>(), std::integral_constant<int, 1>(), 1, 0, 1);
      phase(std::integral_constant<int, NG>(), std::integral_constant<int, 1>(), 0, 1, 1);
      phase(std::integral_constant<int, NR>(), std::integral_constant<int, 2>(), 1, 1, 0);
    } else if constexpr (FORM == kAxis) {
      const float *tx = xt + s * T::kWords * kBW + col;
      int xi[4];
      float ex[T::kE];
#pragma unroll
      for (int k = 0; k < 4; k++) xi[k] = __float_as_int(tx[k * kBW]);
#pragma unroll
      for (int k = 0; k < T::kE; k++) ex[k] = tx[(4 + k) * kBW];
#pragma unroll
      for (int k = 0; k < P; k++) {
        float y[T::kRow];  // the row's cells and factors: the same for every lane
        const float4 *ty = reinterpret_cast<const float4 *>(yt + (s * BH + row0 + k) * T::kRow);
#pragma unroll
        for (int j = 0; j < T::kRow / 4; j++) {
          const float4 t = ty[j];
          y[4 * j] = t.x, y[4 * j + 1] = t.y, y[4 * j + 2] = t.z, y[4 * j + 3] = t.w;
        }
        auto phase = [&](auto N_, Sums<COMP> &a, int ox, int oy, int g) {
          constexpr int N = decltype(N_)::value;
          const float2 *pl = planes + (ox + 2 * oy) * PP + __float_as_int(y[2 * g + oy]) + xi[2 * g + ox];
#pragma unroll
          for (int j = 0; j < N; j++) {
            const float ey = y[4 + 2 * NR * g + N * oy + j];
#pragma unroll
            for (int i = 0; i < N; i++) {
              const float K = fmaxf(fmaf(ex[2 * NR * g + N * ox + i], ey, -L.taper), 0.f);
              a.add(K, pl[j * PW + i]);
            }
          }
        };
        phase(std::integral_constant<int, NR>(), acc[k][0], 0, 0, 0);
        phase(std::integral_constant<int, NG>(), acc[k][1], 1, 0, 1);
        phase(std::integral_constant<int, NG>(), acc[k][1], 0, 1, 1);
        phase(std::integral_constant<int, NR>(), acc[k][2], 1, 1, 0);
      }
    } else {
#pragma unroll
      for (int k = 0; k < P; k++) {
        const int row = row0 + k;
        const int4 an = anchor[s * BH + (row >> 3) * 8 + (col >> 3)];
        const float du = (float)(col & 7), dv = (float)(row & 7);
        const float px = __int_as_float(an.z) + du * Sk.Gf[0] + dv * Sk.Gf[1];
        const float py = __int_as_float(an.w) + du * Sk.Gf[2] + dv * Sk.Gf[3];
        const float flx = floorf(px), fly = floorf(py);
        const int lx = an.x + (int)flx, ly = an.y + (int)fly;
        const float fx = px - flx, fy = py - fly;
        int moved = 0;
        auto phase = [&](auto N_, Sums<COMP> &a, int ox, int oy, int g) {
          constexpr int N = decltype(N_)::value;
          const float hx = L.trunc_k * sg[g] * Sk.hx_unit + 1e-3f, hy = L.trunc_k * sg[g] * Sk.hy_unit + 1e-3f;
          const float unit = sqrtf(log2e * 0.5f) / sg[g];  // K = 2^-(unit |d|)^2 - taper
          float dx, dy;
          const int i0 = first_cell(lx, fx, ox, hx, floorf(0.5f * hx), dx), i = cell_in(i0, PW - N);
          const int j0 = first_cell(ly, fy, oy, hy, floorf(0.5f * hy), dy), j = cell_in(j0, (Sk.box_h >> 1) - N);
          moved |= (i ^ i0) | (j ^ j0);
          const float2 *pl = planes + (ox + 2 * oy) * PP + j * PW + i;
          if constexpr (FORM == kFactored) {
            const float cx = -unit * unit * fmaf(Sk.A[0], Sk.A[0], Sk.A[2] * Sk.A[2]);
            const float cy = -unit * unit * fmaf(Sk.A[1], Sk.A[1], Sk.A[3] * Sk.A[3]);
            float ex[N], ey[N];
#pragma unroll
            for (int c = 0; c < N; c++) {
              const float x = dx + 2.f * (float)c, y = dy + 2.f * (float)c;
              ex[c] = ex2_approx(cx * x * x);
              ey[c] = ex2_approx(cy * y * y);
            }
#pragma unroll
            for (int r = 0; r < N; r++)
#pragma unroll
              for (int c = 0; c < N; c++) {
                const float K = fmaxf(fmaf(ex[c], ey[r], -L.taper), 0.f);
                a.add(K, pl[r * PW + c]);
              }
            return;
          }
          const float2 CX = make_float2(Sk.A[0] * unit, Sk.A[2] * unit), CY = make_float2(Sk.A[1] * unit, Sk.A[3] * unit);
          const float2 DX = make_float2(dx, dx), DY = make_float2(dy, dy);
          const float2 D0 = __ffma2_rn(CY, DY, __fmul2_rn(CX, DX));
          const float2 SX = make_float2(2.f * CX.x, 2.f * CX.y), SY = make_float2(2.f * CY.x, 2.f * CY.y);
#pragma unroll
          for (int r = 0; r < N; r++) {
            float2 D = __ffma2_rn(make_float2((float)r, (float)r), SY, D0);
#pragma unroll
            for (int c = 0; c < N; c++, D = __fadd2_rn(D, SX)) {
              const float K = fmaxf(ex2_approx(-fmaf(D.x, D.x, D.y * D.y)) - L.taper, 0.f);
              a.add(K, pl[r * PW + c]);
            }
          }
        };
        phase(std::integral_constant<int, NR>(), acc[k][0], 0, 0, 0);
        phase(std::integral_constant<int, NG>(), acc[k][1], 1, 0, 1);
        phase(std::integral_constant<int, NG>(), acc[k][1], 0, 1, 1);
        phase(std::integral_constant<int, NR>(), acc[k][2], 1, 1, 0);
        if (moved && u < L.out_w && v0 + row < y_end && abs(lx) < (1 << 20) && abs(ly) < (1 << 20))
          atomicOr(L.status, LPA_ERR_BOUNDS);
      }
    }
  }
  }
  if (u >= L.out_w || (status & LPA_ERR_TIMEOUT)) return;
  // per channel: a pointer to the first row's pixel and the step to the next
  const size_t plane = (size_t)L.out_w * L.out_h, first = (size_t)(v0 + row0) * L.out_w + u;
  const int step = kClasses ? ly : 0;
  const uint32_t next = (uint32_t)L.out_w << step;
  const int rows = v0 + row0 < y_end ? ((y_end - v0 - row0 - 1) >> step) + 1 : 0;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    float val[P];
#pragma unroll
    for (int k = 0; k < P; k++) {
      const float2 a = acc[k][c].value();
      val[k] = a.x > 0.f ? div_approx(a.y, a.x) : __int_as_float(0x7fffffff);
    }
    if (L.out_half) {
      __half *o = reinterpret_cast<__half *>(L.out) + c * plane + first;
#pragma unroll
      for (int k = 0; k < P; k++, o += next)
        if (k < rows) *o = __float2half_rn(val[k]);
    } else {
      float *o = reinterpret_cast<float *>(L.out) + c * plane + first;
#pragma unroll
      for (int k = 0; k < P; k++, o += next)
        if (k < rows) *o = val[k];
    }
    if (L.choice) {
      uint8_t *o = L.choice + c * plane + first;
#pragma unroll
      for (int k = 0; k < P; k++, o += next)
        if (k < rows) *o = acc[k][c].value().x > 0.f ? 0 : 255;
    }
  }
}

// The kernel of plan L for window size (NR, NG), plain (one, two or the most rows per thread) or compensated (two).
template <int NR, int NG, int FORM, bool COMP>
const void *pick_rows(int p) {
  if constexpr (COMP) return (const void *)lpa_mean<NR, NG, FORM, 2, true>;
  else {
    constexpr int kMost = FORM == kPeriodic || FORM == kTabulated ? 8 : 4;
    return p == 1   ? (const void *)lpa_mean<NR, NG, FORM, 1, false>
           : p == 2 ? (const void *)lpa_mean<NR, NG, FORM, 2, false>
                    : (const void *)lpa_mean<NR, NG, FORM, kMost, false>;
  }
}
template <int NR, int NG, bool COMP>
const void *pick(const LpaLaunch &L) {
  return L.mean_k            ? pick_rows<NR, NG, kTabulated, COMP>(L.mean_p)
         : L.mean_lx         ? pick_rows<NR, NG, kPeriodic, COMP>(L.mean_p)
         : L.mean_axis == 1 ? pick_rows<NR, NG, kAxis, COMP>(L.mean_p)
         : L.mean_axis == 2 ? pick_rows<NR, NG, kFactored, COMP>(L.mean_p)
                            : pick_rows<NR, NG, kGeneral, COMP>(L.mean_p);
}

}  // namespace
}  // namespace lpa
