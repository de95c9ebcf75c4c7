// Adaptive windows (CALPA, Sections 5.4-5.5): the steering-matrix pass and the entry points of the
// three passes. The gradient pass (isotropic order-1 green fit) and the steered reconstruction are
// modes of the reconstruction kernel (lpa_kernel.cuh).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "hdr_lpa.h"
#include "lpa_internal.h"
#include "lpa_launch.h"

namespace {

constexpr int kRmax = 10;  // largest radius (output pixels) of the pass-2 disc
constexpr int kBX = 32, kBY = 8;

struct MetricArgs {
  const float2 *grad;
  float *metric;
  int W, H, r;
  int cells;                       // cells of the disc (pixels whose disc lies inside the image)
  int rw[2 * kRmax + 1];           // half width of the disc in row offset dj (|di| <= rw)
  float2 w[2 * kRmax * kRmax + 1];  // Gaussian weight by di^2 + dj^2, as a pair
  double w64[2 * kRmax * kRmax + 1];  // and in FP64
  double scale2;                     // grad_scale^2
  // grad_scale = unit m with unit a power of two (the gradients are staged times it, exactly) and
  // m in [1, 2): T of the scaled gradients is m^2 (a pair) times the sums
  float unit;
  float2 m2;
  float alpha, lambda1, lambda2, min_eig, max_eig;
};

// Pairs of FP32 numbers (x + y unevaluated, |y| <= ulp(x) / 2): about 46 significant bits, from the
// error-free sum (Knuth) and product (FMA residual). An FP64 instruction takes 16 cycles of an SM
// here, a pair operation a handful of FP32 issue slots.
__device__ __forceinline__ float2 pair_norm(float h, float l) {
  const float s = __fadd_rn(h, l);
  return make_float2(s, __fsub_rn(l, __fsub_rn(s, h)));
}
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x), z = __fsub_rn(s, a.x);
  const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, z)), __fsub_rn(b.x, z));
  const float t = __fadd_rn(a.y, b.y), y = __fsub_rn(t, a.y);
  const float f = __fadd_rn(__fsub_rn(a.y, __fsub_rn(t, y)), __fsub_rn(b.y, y));
  const float2 u = pair_norm(s, __fadd_rn(e, t));
  return pair_norm(u.x, __fadd_rn(u.y, f));
}
__device__ __forceinline__ float2 pair_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  return pair_norm(p, fmaf(a.x, b.y, fmaf(a.y, b.x, __fmaf_rn(a.x, b.x, -p))));
}
__device__ __forceinline__ float2 pair_sqrt(float2 a) {  // a >= 0
  if (!(a.x > 0.f)) return make_float2(a.x, 0.f);
  const float s = sqrtf(a.x);
  return pair_norm(s, (__fmaf_rn(-s, s, a.x) + a.y) / (2.f * s));
}

// One thread per output pixel. The gradients of the block and its halo are staged in shared
// memory as the products gx^2, gx gy, gy^2, each an exact FP32 pair, and T = sum_i w_i g_i g_i^T
// over the disc is summed in pairs: T of a straight edge is nearly rank one, and its small
// eigenvalue is the difference of large sums. The eigenvalues l1,2 = h +- sqrt(((a - c) / 2)^2 + b^2)
// and the components of the eigenvector of l1 ((b, l1 - a) or (l1 - c, b), the longer) are formed in
// pairs too; what follows them (square roots, the direction's normalisation, elongation, the power
// and the matrix) has no cancellation and runs in FP32.
//
// Bound by the FP32 pipe: 36 pipe cycles per warp and weighted term (12 operations on each of three
// sums, gx^2 and gy^2 side by side in paired instructions). The same sums in FP64 kept the FP64
// pipe 84 % busy: gradients and matrices of 1920 x 1080 with 29 cells took 751 us, with this kernel
// and looped discs 324 us.
//
// UNIT: the disc of window_sigma 1 (radius 3: half widths 0, 2, 2, 3, 2, 2, 0). The Gaussian factors, so the
// rows of a 32 x 16 block are summed along x first (over half widths 2 and 3, into shared memory) and
// those sums along y: 7 weighted terms a pixel instead of 28 (gradients and matrices of 1920 x 1080: 212 us
// with the 29 cells unrolled, 183 us so, 179 with cells of equal weight added first). Four CTAs per SM at 47 KB and 64 registers.
constexpr int kUnitBY = 16, kUnitR = 3;
__host__ __device__ constexpr int unit_row(int dj) { return dj == 0 ? 3 : dj == 3 || dj == -3 ? 0 : 2; }

// T's sums in pairs: (sum w gx^2, sum w gy^2) and sum w gx gy, with what rounding dropped.
struct DiscSum {
  float2 S, E;
  float s, e;
  __device__ __forceinline__ DiscSum() : S(make_float2(0.f, 0.f)), E(make_float2(0.f, 0.f)), s(0.f), e(0.f) {}
  __device__ __forceinline__ DiscSum(float4 d, float2 x) : S(make_float2(d.x, d.y)), E(make_float2(d.z, d.w)), s(x.x), e(x.y) {}
  __device__ __forceinline__ void add(float2 w, float4 d, float2 x) {
    const float2 minus = make_float2(-1.f, -1.f);
    {
      const float2 X = make_float2(d.x, d.y), W = make_float2(w.x, w.x);
      const float2 P = __fmul2_rn(W, X);
      float2 q = __ffma2_rn(W, X, make_float2(-P.x, -P.y));
      q = __ffma2_rn(W, make_float2(d.z, d.w), q);
      q = __ffma2_rn(make_float2(w.y, w.y), X, q);
      const float2 t = __fadd2_rn(S, P), z = __ffma2_rn(S, minus, t);
      const float2 k = __ffma2_rn(__ffma2_rn(z, minus, t), minus, S);  // S - (t - z)
      E = __fadd2_rn(E, __fadd2_rn(__fadd2_rn(k, __ffma2_rn(z, minus, P)), q));
      S = t;
    }
    {
      const float p = __fmul_rn(w.x, x.x);
      const float q = fmaf(w.y, x.x, fmaf(w.x, x.y, __fmaf_rn(w.x, x.x, -p)));
      const float t = __fadd_rn(s, p), z = __fsub_rn(t, s);
      const float k = __fsub_rn(s, __fsub_rn(t, z));
      e = __fadd_rn(e, __fadd_rn(__fadd_rn(k, __fsub_rn(p, z)), q));
      s = t;
    }
  }
  // Two terms of one weight: added first (an error-free sum and what it dropped), then weighted once.
  __device__ __forceinline__ void add(float2 w, float4 da, float2 xa, float4 db, float2 xb) {
    const float2 minus = make_float2(-1.f, -1.f), A = make_float2(da.x, da.y), B = make_float2(db.x, db.y);
    const float2 t = __fadd2_rn(A, B), z = __ffma2_rn(A, minus, t);
    const float2 k = __fadd2_rn(__ffma2_rn(__ffma2_rn(z, minus, t), minus, A), __ffma2_rn(z, minus, B));
    const float2 l = __fadd2_rn(__fadd2_rn(make_float2(da.z, da.w), make_float2(db.z, db.w)), k);
    const float x = __fadd_rn(xa.x, xb.x), y = __fsub_rn(x, xa.x);
    const float m = __fadd_rn(__fsub_rn(xa.x, __fsub_rn(x, y)), __fsub_rn(xb.x, y));
    add(w, make_float4(t.x, t.y, l.x, l.y), make_float2(x, __fadd_rn(__fadd_rn(xa.y, xb.y), m)));
  }
  __device__ __forceinline__ float4 d() const { return make_float4(S.x, S.y, E.x, E.y); }
  __device__ __forceinline__ float2 x() const { return make_float2(s, e); }
};

// The eigenvalues of T and the steering matrix of pixel (u, v).
__device__ __forceinline__ void store_matrix(const MetricArgs &A, int r, const DiscSum &D, int u, int v) {
  const float2 S = D.S, E = D.E;
  const float s = D.s, e = D.e;
  int M = A.cells;
  if (u < r || v < r || u + r >= A.W || v + r >= A.H) {  // disc cells inside the image
    M = 0;
    for (int dj = -r; dj <= r; dj++) {
      const int rw = A.rw[dj + r];
      if (v + dj >= 0 && v + dj < A.H) M += min(u + rw, A.W - 1) - max(u - rw, 0) + 1;
    }
  }
  // T brought to [1, 2) by a power of two, so that the squares below neither overflow nor underflow
  const int et = min(max((__float_as_int(fmaxf(S.x, S.y)) >> 23) & 255, 1), 253);
  const float up = __int_as_float(et << 23), down = __int_as_float((254 - et) << 23);
  const float2 a = pair_mul(pair_norm(S.x * down, E.x * down), A.m2);
  const float2 c = pair_mul(pair_norm(S.y * down, E.y * down), A.m2);
  const float2 b = pair_mul(pair_norm(s * down, e * down), A.m2);
  const float2 sum = pair_add(a, c), dif = pair_add(a, pair_neg(c));
  const float2 h = make_float2(0.5f * sum.x, 0.5f * sum.y), t = make_float2(0.5f * dif.x, 0.5f * dif.y);
  const float2 d = pair_sqrt(pair_add(pair_mul(t, t), pair_mul(b, b)));
  const float2 l1 = pair_add(h, d), l2 = pair_add(h, pair_neg(d));
  // the eigenvector of l1 in its longer form: |l1 - c| > |l1 - a| where a > c
  const bool wide = dif.x > 0.f;
  const float2 Ux = wide ? pair_add(l1, pair_neg(c)) : b, Uy = wide ? b : pair_add(l1, pair_neg(a));
  float ux = Ux.x, uy = Uy.x;
  float L1 = l1.x * up, L2 = fmaxf(l2.x, 0.f) * up;
  if (!(l2.x >= 0x1p-18f * l1.x)) {
    if (l1.x <= 3.402823466e38f) {
      // Nearly rank one: the pairs hold l2 to about 2^-45 l1, less than an FP32 value needs below this ratio (noise keeps
      // it above in camera frames; clean edges and ramps, and lone gradients, are below). Their eigenvector is good to
      // 2^-44 all the same, so l2 is summed again as w (g . v)^2 over the disc, v across it: g . v from exact products,
      // no cancellation after it. 1920 x 1080 clean gradients with the default disc: 0.13 ms; FP64 sums there 1.37 ms (0.55 ms
      // where every pixel is summed in FP64, from staged products), and these hold l2 to 2^-52 l1 only.
      const int eh = (127 - et) >> 1;
      const float half = __int_as_float((127 + eh) << 23), back = __int_as_float((127 - eh) << 23);
      float sum = 0.f, rest = 0.f;  // and what its additions rounded away
      for (int dj = max(-r, -v); dj <= min(r, A.H - 1 - v); dj++) {
        const int rw = A.rw[dj + r];
        const float2 *row = A.grad + (size_t)(v + dj) * A.W + u;
        for (int di = max(-rw, -u); di <= min(rw, A.W - 1 - u); di++) {
          const float2 g = row[di];
          const float gx = g.x * A.unit * half, gy = g.y * A.unit * half;
          const float px = __fmul_rn(gy, Ux.x), py = __fmul_rn(gx, Uy.x);
          const float low = (__fmaf_rn(gy, Ux.x, -px) - __fmaf_rn(gx, Uy.x, -py)) + (gy * Ux.y - gx * Uy.y);
          const float q = __fadd_rn(__fsub_rn(px, py), low);
          const float term = A.w[di * di + dj * dj].x * q * q, next = __fadd_rn(sum, term);
          rest += __fsub_rn(term, __fsub_rn(next, sum));
          sum = next;
        }
      }
      L2 = (sum + rest) / fmaf(ux, ux, uy * uy) * A.m2.x * back * back;
    } else {
      // sums, or products with the scale, that left FP32's range: in FP64 from the gradients
      double da = 0.0, db = 0.0, dc = 0.0;
      for (int dj = max(-r, -v); dj <= min(r, A.H - 1 - v); dj++) {
        const int rw = A.rw[dj + r];
        const float2 *row = A.grad + (size_t)(v + dj) * A.W + u;
        for (int di = max(-rw, -u); di <= min(rw, A.W - 1 - u); di++) {
          const float2 g = row[di];
          const double w = A.w64[di * di + dj * dj], gx = g.x, gy = g.y;
          da = fma(w, gx * gx, da);
          db = fma(w, gx * gy, db);
          dc = fma(w, gy * gy, dc);
        }
      }
      da *= A.scale2;
      db *= A.scale2;
      dc *= A.scale2;
      const double dh = 0.5 * (da + dc), dd = sqrt(0.25 * (da - dc) * (da - dc) + db * db);
      L1 = (float)(dh + dd);
      L2 = (float)fmax(dh - dd, 0.0);
      const double vx = da > dc ? dh + dd - dc : db, vy = da > dc ? db : dh + dd - da;
      // into FP32's range before the conversion, by a power of two
      const int vexp = (__double2hiint(fmax(fabs(vx), fabs(vy))) >> 20) & 2047;
      const double vunit = __hiloint2double(min(max(2046 - vexp, 1), 2046) << 20, 0);
      ux = (float)(vx * vunit);
      uy = (float)(vy * vunit);
    }
  }
  const int ex = (__float_as_int(fmaxf(fabsf(ux), fabsf(uy))) >> 23) & 255;  // its exponent removed, exactly
  const float unit = __int_as_float(min(max(253 - ex, 1), 254) << 23);
  ux *= unit;
  uy *= unit;
  const float n2 = ux * ux + uy * uy;
  if (n2 == 0.f) {  // T = 0
    ux = 1.f;
    uy = 0.f;
  } else {
    const float nrm = sqrtf(n2);
    ux /= nrm;
    uy /= nrm;
  }
  const float s1 = sqrtf(L1), s2 = sqrtf(L2);
  const float elong = (s1 + A.lambda1) / (s2 + A.lambda1);
  const float gamma = powf((s1 * s2 + A.lambda2) / (float)M, A.alpha);
  const float ea = fminf(fmaxf(gamma * elong, A.min_eig), A.max_eig);  // along u1: across the edge
  const float eb = fminf(fmaxf(gamma / elong, A.min_eig), A.max_eig);  // along u2: along the edge
  float *o = A.metric + ((size_t)v * A.W + u) * 3;
  o[0] = ea * ux * ux + eb * uy * uy;
  o[1] = (ea - eb) * ux * uy;
  o[2] = ea * uy * uy + eb * ux * ux;
}

template <bool UNIT>
__global__ void __launch_bounds__(kBX *kBY, UNIT ? 4 : 1) calpa_metric(const __grid_constant__ MetricArgs A) {
  extern __shared__ __align__(16) float4 sm[];
  constexpr int BY = UNIT ? kUnitBY : kBY;
  const int r = UNIT ? kUnitR : A.r, TW = kBX + 2 * r, TH = BY + 2 * r;
  float4 *sd = sm;                                        // (gx^2, gy^2, their residuals)
  float2 *sx = reinterpret_cast<float2 *>(sm + TW * TH);  // (gx gy, its residual)
  // one-dimensional grid over the blocks (any output height)
  const int nbx = (A.W + kBX - 1) / kBX;
  const int bx0 = (int)(blockIdx.x % nbx) * kBX, by0 = (int)(blockIdx.x / nbx) * BY;
  for (int ty = threadIdx.y; ty < TH; ty += kBY) {
    const int Y = by0 - r + ty;
    const float2 *row = A.grad + (size_t)max(Y, 0) * A.W;
    for (int tx = threadIdx.x; tx < TW; tx += kBX) {
      const int X = bx0 - r + tx;
      float2 g = (X >= 0 && X < A.W && Y >= 0 && Y < A.H) ? row[X] : make_float2(0.f, 0.f);
      g = make_float2(g.x * A.unit, g.y * A.unit);
      const float xx = __fmul_rn(g.x, g.x), yy = __fmul_rn(g.y, g.y), xy = __fmul_rn(g.x, g.y);
      sd[ty * TW + tx] = make_float4(xx, yy, __fmaf_rn(g.x, g.x, -xx), __fmaf_rn(g.y, g.y, -yy));
      sx[ty * TW + tx] = make_float2(xy, __fmaf_rn(g.x, g.y, -xy));
    }
  }
  __syncthreads();
  const int u = bx0 + threadIdx.x, mid = threadIdx.x + r;
  if constexpr (UNIT) {
    constexpr int H = kUnitBY + 2 * kUnitR - 2;  // rows from the second staged one to the last but one
    float4 *d2 = reinterpret_cast<float4 *>(sx + TW * TH), *d3 = d2 + H * kBX;  // row sums over |di| <= 2, <= 3
    float2 *x2 = reinterpret_cast<float2 *>(d3 + kUnitBY * kBX), *x3 = x2 + H * kBX;
    const float2 w1 = A.w[1], w4 = A.w[4], w9 = A.w[9];
#pragma unroll 1
    for (int y = threadIdx.y; y < H; y += kBY) {
      const int at = (y + 1) * TW + mid, to = y * kBX + threadIdx.x;
      DiscSum a(sd[at], sx[at]);
      a.add(w1, sd[at - 1], sx[at - 1], sd[at + 1], sx[at + 1]);
      a.add(w4, sd[at - 2], sx[at - 2], sd[at + 2], sx[at + 2]);
      d2[to] = a.d();
      x2[to] = a.x();
      if (y < kUnitR - 1 || y > H - kUnitR) continue;
      a.add(w9, sd[at - 3], sx[at - 3], sd[at + 3], sx[at + 3]);
      d3[to - (kUnitR - 1) * kBX] = a.d();
      x3[to - (kUnitR - 1) * kBX] = a.x();
    }
    __syncthreads();
#pragma unroll 1
    for (int y = threadIdx.y; y < kUnitBY; y += kBY) {
      const int at = (y + kUnitR - 1) * kBX + threadIdx.x, up = y * TW + mid, dn = up + 2 * kUnitR * TW;
      DiscSum a(d3[y * kBX + threadIdx.x], x3[y * kBX + threadIdx.x]);
      a.add(w1, d2[at - kBX], x2[at - kBX], d2[at + kBX], x2[at + kBX]);
      a.add(w4, d2[at - 2 * kBX], x2[at - 2 * kBX], d2[at + 2 * kBX], x2[at + 2 * kBX]);
      a.add(w9, sd[up], sx[up], sd[dn], sx[dn]);
      if (u < A.W && by0 + y < A.H) store_matrix(A, kUnitR, a, u, by0 + y);
    }
  } else {
    const int v = by0 + threadIdx.y;
    if (u >= A.W || v >= A.H) return;
    DiscSum a;
    for (int dj = -r; dj <= r; dj++) {
      const int rw = A.rw[dj + r], at = (threadIdx.y + r + dj) * TW + mid;
#pragma unroll 2
      for (int di = -rw; di <= rw; di++) a.add(A.w[di * di + dj * dj], sd[at + di], sx[at + di]);
    }
    store_matrix(A, r, a, u, v);
  }
}

hdr_status check_calpa(const hdr_calpa_params *c) {
  if (!c) return lpa_fail(HDR_E_INVALID, "calpa is NULL");
  auto fin = [](double x) { return std::isfinite(x); };
  if (!(c->grad_sigma > 0.0) || !fin(c->grad_sigma))
    return lpa_fail(HDR_E_INVALID, "grad_sigma must be finite and > 0");
  if (!(c->window_sigma > 0.0) || !(3.0 * c->window_sigma < kRmax + 1.0))
    return lpa_fail(HDR_E_INVALID, "window_sigma must be > 0 with 3 window_sigma < 11");
  // bounds keep every FP32 quantity of the matrix pass inside the normal range
  if (!(c->alpha >= 0.0) || !(c->alpha <= 4.0)) return lpa_fail(HDR_E_INVALID, "alpha must be in [0, 4]");
  if (!(c->lambda1 >= 1e-6 && c->lambda1 <= 1e6) || !(c->lambda2 >= 1e-12 && c->lambda2 <= 1e12))
    return lpa_fail(HDR_E_INVALID, "lambda1 in [1e-6, 1e6] and lambda2 in [1e-12, 1e12] required");
  if (!(c->min_eig >= 1e-6) || !(c->max_eig >= c->min_eig) || !(c->max_eig <= 1e6))
    return lpa_fail(HDR_E_INVALID, "1e-6 <= min_eig <= max_eig <= 1e6 required");
  if (!(c->grad_scale > 0.0) || !(c->grad_scale <= 1e6)) return lpa_fail(HDR_E_INVALID, "grad_scale must be in (0, 1e6]");
  return HDR_OK;
}

}  // namespace

hdr_status lpa_check_calpa(const hdr_calpa_params *c) { return check_calpa(c); }

double lpa_calpa_reach(const hdr_calpa_params *calpa) { return 1.0 / std::sqrt(calpa->min_eig); }

namespace {
// Pass 1: one isotropic order-1 fit at grad_sigma (ahead: see lpa_launch_mode).
hdr_status gradients(hdr_ctx *ctx, int32_t rig_id, const hdr_params *params, const hdr_calpa_params *calpa,
                     const uint16_t *const *raw_dev, float *grad_dev, cudaStream_t st, bool ahead) {
  hdr_status s = check_calpa(calpa);
  if (s) return s;
  if (!params) return lpa_fail(HDR_E_INVALID, "params is NULL");
  hdr_params p = *params;
  p.order = 1;
  p.n_scales = 1;
  p.sigma[0] = calpa->grad_sigma;
  return lpa_launch_mode(ctx, rig_id, &p, raw_dev, LPA_GRADIENTS, grad_dev, 1.0, nullptr, nullptr, st, ahead);
}
}  // namespace

hdr_status lpa_calpa_prepare(hdr_ctx *ctx, int32_t rig_id, const hdr_params *params, const hdr_calpa_params *calpa,
                             const uint16_t *const *raw_dev, float *scratch, cudaStream_t st) {
  const size_t npx = (size_t)params->out_w * params->out_h;
  if (npx == 0) return HDR_OK;
  float *grad = scratch, *metric = scratch + npx * 2;
  // inside a batch, whose plans may point into the context's conversion buffer: the pass converts
  // its footprints itself
  hdr_status s = gradients(ctx, rig_id, params, calpa, raw_dev, grad, st, false);
  if (s) return s;
  return hdr_calpa_metric(ctx, params->out_w, params->out_h, calpa, grad, metric, st);
}

extern "C" {

void hdr_calpa_params_default(hdr_calpa_params *c) {
  if (!c) return;
  c->grad_sigma = 1.2;
  c->window_sigma = 1.0;
  c->alpha = 0.3;
  c->lambda1 = 1.0;
  c->lambda2 = 1e-3;
  c->min_eig = 0.25;
  c->max_eig = 16.0;
  c->grad_scale = 0.1;
}

hdr_status hdr_calpa_gradients(hdr_ctx *ctx, int32_t rig_id, const hdr_params *params, const hdr_calpa_params *calpa,
                               const uint16_t *const *raw_dev, float *grad_dev, void *cuda_stream) {
  return gradients(ctx, rig_id, params, calpa, raw_dev, grad_dev, (cudaStream_t)cuda_stream, true);
}

hdr_status hdr_calpa_metric(hdr_ctx *ctx, int32_t out_w, int32_t out_h, const hdr_calpa_params *calpa,
                            const float *grad_dev, float *metric_dev, void *cuda_stream) {
  if (!ctx) return lpa_fail(HDR_E_INVALID, "ctx is NULL");
  hdr_status st = check_calpa(calpa);
  if (st) return st;
  if (out_w < 0 || out_h < 0) return lpa_fail(HDR_E_INVALID, "negative output size");
  if ((long long)out_w * out_h > (1LL << 31) / 4) return lpa_fail(HDR_E_UNSUPPORTED, "output too large");
  if ((long long)out_w * out_h == 0) return HDR_OK;
  if (!grad_dev || !metric_dev) return lpa_fail(HDR_E_INVALID, "grad_dev and metric_dev are required");
  if (reinterpret_cast<uintptr_t>(grad_dev) % 8) return lpa_fail(HDR_E_INVALID, "grad_dev not 8-byte aligned");
  if (cudaSetDevice(lpa_ctx_device(ctx)) != cudaSuccess) return lpa_fail(HDR_E_CUDA, "cudaSetDevice failed");
  MetricArgs A{};
  A.grad = reinterpret_cast<const float2 *>(grad_dev);
  A.metric = metric_dev;
  A.W = out_w;
  A.H = out_h;
  const double ws = calpa->window_sigma, R = 3.0 * ws;
  A.r = (int)std::floor(R);
  for (int dj = -A.r; dj <= A.r; dj++) {
    int rw = 0;
    while (rw + 1 <= A.r && (double)((rw + 1) * (rw + 1) + dj * dj) <= R * R) rw++;
    A.rw[dj + A.r] = rw;
  }
  auto pair = [](double x) { return make_float2((float)x, (float)(x - (double)(float)x)); };
  A.cells = 0;
  for (int dj = -A.r; dj <= A.r; dj++) A.cells += 2 * A.rw[dj + A.r] + 1;
  for (int k = 0; k <= 2 * A.r * A.r; k++) A.w[k] = pair(A.w64[k] = std::exp(-(double)k / (2.0 * ws * ws)));
  A.scale2 = calpa->grad_scale * calpa->grad_scale;
  A.unit = (float)std::ldexp(1.0, std::max(std::ilogb(calpa->grad_scale), -100));
  const double m = calpa->grad_scale / (double)A.unit;
  A.m2 = pair(m * m);
  A.alpha = (float)calpa->alpha;
  A.lambda1 = (float)calpa->lambda1;
  A.lambda2 = (float)calpa->lambda2;
  A.min_eig = (float)calpa->min_eig;
  A.max_eig = (float)calpa->max_eig;
  bool unit = A.r == kUnitR;
  for (int dj = -kUnitR; dj <= kUnitR && unit; dj++) unit = A.rw[dj + kUnitR] == unit_row(dj);
  const int by = unit ? kUnitBY : kBY;
  const unsigned blocks = (unsigned)(((long long)out_w + kBX - 1) / kBX * (((long long)out_h + by - 1) / by));
  size_t px = (size_t)(kBX + 2 * A.r) * (by + 2 * A.r);          // at most 35 KB
  if (unit) px += (size_t)kBX * (2 * kUnitBY + 2 * kUnitR - 2);  // and the row sums: 46.6 KB
  const size_t smem = px * (sizeof(float4) + sizeof(float2));
  if (unit) calpa_metric<true><<<blocks, dim3(kBX, kBY), smem, (cudaStream_t)cuda_stream>>>(A);
  else calpa_metric<false><<<blocks, dim3(kBX, kBY), smem, (cudaStream_t)cuda_stream>>>(A);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return lpa_fail(HDR_E_CUDA, cudaGetErrorString(e));
  return HDR_OK;
}

hdr_status hdr_reconstruct_steered(hdr_ctx *ctx, int32_t rig_id, const hdr_params *params,
                                   const hdr_calpa_params *calpa, const uint16_t *const *raw_dev,
                                   const float *metric_dev, void *out_dev, uint8_t *choice_dev, void *cuda_stream) {
  hdr_status st = check_calpa(calpa);
  if (st) return st;
  if (!params) return lpa_fail(HDR_E_INVALID, "params is NULL");
  if (!metric_dev && (long long)params->out_w * params->out_h > 0) return lpa_fail(HDR_E_INVALID, "metric_dev is NULL");
  return lpa_launch_mode(ctx, rig_id, params, raw_dev, LPA_STEERED, const_cast<float *>(metric_dev),
                         lpa_calpa_reach(calpa), out_dev, choice_dev, (cudaStream_t)cuda_stream, true);
}

hdr_status hdr_reconstruct_adaptive(hdr_ctx *ctx, int32_t rig_id, const hdr_params *params,
                                    const hdr_calpa_params *calpa, const uint16_t *const *raw_dev, void *out_dev,
                                    uint8_t *choice_dev, void *cuda_stream) {
  if (!ctx) return lpa_fail(HDR_E_INVALID, "ctx is NULL");
  hdr_status st = check_calpa(calpa);
  if (st) return st;
  st = lpa_check_params(params);
  if (st) return st;
  const size_t npx = (size_t)params->out_w * params->out_h;
  if (npx == 0) return HDR_OK;
  void *scratch = nullptr;
  st = lpa_ctx_calpa_scratch(ctx, npx * 5 * sizeof(float), &scratch);
  if (st) return st;
  float *grad = static_cast<float *>(scratch), *metric = grad + npx * 2;
  st = hdr_calpa_gradients(ctx, rig_id, params, calpa, raw_dev, grad, cuda_stream);
  if (st) return st;
  st = hdr_calpa_metric(ctx, params->out_w, params->out_h, calpa, grad, metric, cuda_stream);
  if (st) return st;
  return hdr_reconstruct_steered(ctx, rig_id, params, calpa, raw_dev, metric, out_dev, choice_dev, cuda_stream);
}

}  // extern "C"
