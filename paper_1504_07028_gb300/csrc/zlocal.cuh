// z-update (12) of SegSALSA-STR in the pixel domain, one launch: z = (3 I + J^T J)^{-1} rhs.
//
// With weights normalised as the method's Gaussian ones (c = sum_j omega_j^2 = 1, or less) the 5-point
// operator A = d - c (S_x + S_x^{-1} + S_y + S_y^{-1}), d = 3 + 4c, is so well conditioned
// (eigenvalues in [3, 3 + 8c]) that its inverse is local: it decays by 0.209 or less per
// pixel, and the Chebyshev semi-iteration (Golub and Varga) on the Jacobi splitting
//   x_{k+1} = w_{k+1} (g (sum of the 4 neighbours of x_k) + b) + (1 - w_{k+1}) x_{k-1},
//   g = c / d, b = rhs / d, w_1 = 1, w_2 = 2 / (2 - r^2), w_{k+1} = 1 / (1 - r^2 w_k / 4), r = 4g,
// contracts the error by s = r / (1 + sqrt(1 - r^2)) <= 0.314 a step: 17 steps from x_0 = 0 leave
// at most 2 s^17 = 6e-9 of it, below half an FP32 unit. The 5-point graph is bipartite, so
// (cyclic form) a step updates only the points of one colour, in place. Measured against 64 bits
// on random fields: 5.1e-8 relative, where the row transforms and column recursions of fft.cuh,
// which every other case takes (FP64, larger weights), leave 1.8e-7.
//
// A strip is computed from its pixels and a halo of ZL_HALO. What lies beyond counts as 0, except at
// the first and last column of the streaming form, whose missing neighbour is replaced by a value of
// the same lane's four columns (a shuffle past the end of the warp returns it): either way a neighbour off
// by at most twice the field's largest value, of which 0.209^12 = 7e-9 reaches the wanted pixels.
// Nothing depends on the image's size: no transform length, no period (halo pixels wrap), any
// class count.
#pragma once

#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace sgs {

constexpr int ZL_HALO = 12;
constexpr int ZL_STEPS = 17;
constexpr int ZL_EARLY = 2;          // steps 2 and 3 with their own weights; then the limit weight
constexpr int ZL_WIDTH = 128;        // columns of a strip with its halo
constexpr double ZL_MAX_C = 1.0005;  // largest sum of squared weights (17 steps are enough up to here)

// Step coefficients: x <- cw * (neighbour sum) + c1 * x + cb * bs, bs = (w_limit / d) rhs. Steps
// 4 .. 17 take the limit weight (w_4 - w_limit < 1e-3; the error bound grows from 1.3e-8 to 1.5e-8).
struct ZlCoef {
  float bs;              // w_limit / d
  float2 b0;             // 1 / w_limit (twice): the first step, x = b
  float2 cw[ZL_EARLY + 1], c1[ZL_EARLY + 1], cb[ZL_EARLY];  // [ZL_EARLY]: the limit weight (cb = 1)
};

inline ZlCoef zl_coef(double c) {
  ZlCoef q{};
  auto two = [](double v) { return make_float2((float)v, (float)v); };
  const double d = 3.0 + 4.0 * c, g = c / d, r = 4.0 * g;
  const double wl = 2.0 / (1.0 + std::sqrt(1.0 - r * r));
  q.bs = (float)(wl / d);
  q.b0 = two(1.0 / wl);
  double w = 2.0 / (2.0 - r * r);
  for (int i = 0; i < ZL_EARLY; ++i) {
    q.cw[i] = two(w * g);
    q.c1[i] = two(1.0 - w);
    q.cb[i] = two(w / wl);
    w = 1.0 / (1.0 - 0.25 * r * r * w);
  }
  q.cw[ZL_EARLY] = two(wl * g);
  q.c1[ZL_EARLY] = two(1.0 - wl);
  return q;
}

constexpr int ZB_ROWS = 4;           // rows of a thread's block in the block form
constexpr int ZB_THREADS = 640;      // largest CTA of the block form
constexpr int ZB_MAXSIDE = 256;      // longest tile side with its halo

// Work split. kc = 0, the streaming form: nx strips, ny segments. kc = 1, 2, 4, the block form:
// nx x ny tiles of nbx x nby thread blocks (with the halo), kc classes a CTA.
struct ZlPlan {
  int nx, ny;
  int kc, nbx, nby, threads;
};
// Shared memory of a block-form CTA: the tile's rhs planes, then (in their place) the edges.
inline size_t zb_smem(const ZlPlan& p) {
  const size_t planes = (size_t)p.kc * (4 * p.nbx * ZB_ROWS * p.nby + 4) * 4;
  const size_t edges = (size_t)(p.threads + 1) * 2 * 32;
  return std::max(planes, edges);
}

struct ZlArgs {
  int H, W, K, ng;       // ng: class quads
  ZlPlan p;
  const float* src;      // dense rhs [n][K], or nullptr: the sweep's tile partials
  const float* P;        // [tiles][ng][EHmax][EWmax][4]
  int ntx, EHmax, EWmax;
  const int* offY;       // [H][2]: offset of a row's covers in P, in quads, at tile column 0; -1: absent
  const int* covX;       // [W][2]: (tile column << 16 | column in the tile), -1 when absent
  float* z;
  ZlCoef q;
};

// Work split of the smaller modelled time (us on one GB300; the constants fit event times of both
// forms over 64 x 64, K = 4 to 2048 x 2048, K = 16). Streaming: two CTAs an SM, 0.45 us a row with
// both at work and 0.38 us alone, a segment of h rows taking h + 28 of them. Block form: one CTA
// an SM, 3.5 us and 0.0065 us a thread (more where only one class of a quad is loaded). The model has
// one image on an idle GPU in mind; the images of a batch, which share it, take the same split
// all the same, because each has to match its own handle bit for bit and results depend on the split.
inline ZlPlan zl_plan(int H, int W, int K) {
  const int sms = 152, edge = 2 * ZL_HALO, useful = ZL_WIDTH - edge;
  ZlPlan p{(W + useful - 1) / useful, 1, 0, 0, 0, 128};
  const long long cols = (long long)p.nx * ((K + 3) / 4);
  double best = 1e300;
  for (int ny = 1; ny <= H && cols * (ny - 1) <= 16 * sms; ++ny) {
    const double rows = (H + ny - 1) / ny + edge + ZL_STEPS - ZL_HALO - 1;
    const long long waves = (cols * ny + 2 * sms - 1) / (2 * sms);
    const double cost = waves * (3.0 + rows * (cols * ny > sms ? 0.45 : 0.38));
    if (cost < best) { best = cost; p.ny = ny; }
  }
  const int least = edge / 4 + 1, most = ZB_MAXSIDE / 4;
  for (int kc = 1; kc <= 4 && kc < 2 * K; kc *= 2) {
    const int ngc = (K + kc - 1) / kc;
    for (int mx = least; mx <= most && mx * least * kc <= ZB_THREADS; ++mx) {
      const int nx = (W + 4 * mx - edge - 1) / (4 * mx - edge);
      const int nbx = ((W + nx - 1) / nx + edge + 3) / 4;
      if (nbx < mx) continue;                    // the same split as a narrower tile's
      for (int my = least; my <= most && nbx * my * kc <= ZB_THREADS; ++my) {
        const int ny = (H + ZB_ROWS * my - edge - 1) / (ZB_ROWS * my - edge);
        const int nby = ((H + ny - 1) / ny + edge + ZB_ROWS - 1) / ZB_ROWS;
        if (nby < my) continue;
        const int thr = (nbx * nby * kc + 31) / 32 * 32;
        const long long waves = ((long long)nx * ny * ngc + sms - 1) / sms;
        const double cost = waves * (3.5 + 0.0065 * thr * (kc == 1 ? (K > 4 ? 1.8 : 1.2) : 1.0));
        if (cost < best) { best = cost; p = ZlPlan{nx, ny, kc, nbx, nby, thr}; }
      }
    }
  }
  return p;
}

cudaError_t launch_zlocal(const ZlArgs& a, cudaStream_t st);

}  // namespace sgs
