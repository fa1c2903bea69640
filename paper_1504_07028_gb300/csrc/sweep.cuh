// Fused SALSA sweep (u-update (13) + d-update (14) + right-hand side of the next z-update (12))
// for SegSALSA-STR, one launch per iteration.
//
// Per pixel i (Sec. 4):
//   v1 = z - d1,  v2 = J z - d2,  v3 = z - d3,  v4 = z - d4              (G z^{k+1} - d^k)
//   u1 = prox of -ln(p^T .)/mu at v1 (positive root of s^2 - (p^T v1) s - |p|^2/mu = 0)
//   u2 = Schatten-p prox of (lambda/mu)||.||_{S_p} at the (L K) x 2 matrix v2  (Sec. 3-4)
//   u3 = max(v3, 0);   u4 = v4 - (1^T v4 - 1)/K                          (MPOs of g3, g4)
//   d_j <- u_j - v_j  (= d_j - (G z - u_j), eq. 14)
//   rhs = (u1 + d1) + J^T (u2 + d2) + (u3 + d3) + (u4 + d4)              (G^T (u + d), eq. 12)
//
// Work mapping. A CTA owns a tile of pixels (balanced tiling of the image) and NT = 256 threads,
// or 64 where the image has fewer than 152 tiles of 256: NC <= NT / G columns x G lanes. The G
// lanes of a column hold the classes of one pixel (class
// k = lane), so the 2x2 Gram matrix [Jz]_i^T [Jz]_i of eq. (5) is a G-lane shuffle sum and
// each lane keeps its 2L Jacobian entries in registers. Each column walks down the tile rows.
// The Jacobian stencil reads z from a shared-memory copy of the tile plus its halo
// ([-M, M+1] around every pixel). J^T w is a scatter: pixel i sends +/- omega_j w to the
// (2M+2)^2 neighbours i + s_j (+ e_h / e_v). Each thread keeps those sums for the rows it can
// still touch in a (2M+2)x(2M+2) register window; every row step, the finished top window row
// goes through exclusive shared-memory slots, is summed in a fixed order by the owner of each
// column and stored as one row of the tile's partials P (tile plus halo). The z-update (the
// pixel-domain kernels of zlocal.cu, or the row transforms of fft.cuh) adds the overlapping tiles
// when it reads rhs (no atomics anywhere: deterministic).
#pragma once

#include "common.cuh"
#include "giveup.h"

namespace sgs {

template <typename T>
struct SweepArgs {
  int H, W, K;
  int NC;                // columns per tile (<= threads / G)
  int ntx, nty;          // tile grid
  int EHmax, EWmax;      // extents of the P tile slots (tile + halo), in pixels
  const T* z;            // [n][K]
  const T* p;            // [n][K]
  T* dloc;               // [n][3][K]  (d1, d3, d4): full form of the local duals
  T* dcmp;               // [n][K + 2] (d3, c1, c4): compact form, d1 = c1 p, d4 = c4 1 (affine g4)
  int cin;               // affine g4: the local duals come in compact form (else full form);
                         // the affine sweep writes the compact form, the simplex sweep the full
  T* d2;                 // [n][L][K][2]
  T* d2o;                // the new d2 (d2 itself: in place)
  T* dloco;              // simplex: the new full form (dloc itself: in place)
  T* P;                  // per tile: partial sums of G^T(u + d) over [EHmax][EWmax] pixels; class k of
                         // pixel q at q * pstr + (k / 4) * pquad + k % 4 of the tile's ptile values
  int pstr, pquad, ptile;  // K, 4, EHmax EWmax K: pixel-major; 4, 4 EHmax EWmax, ...: planes of
                           // four classes (the z-update of zlocal.cuh reads whole quads)
  T* P2;                 // DIAG: partial sums of G^T d (dual residual), [tiles][EHmax][EWmax][K]
  double* diag_sq;       // DIAG: per tile sum of squared dual changes (primal residual)
  const T* omega;        // [L] shift weights
  T tau;                 // lambda / mu
  T mu;
  T invK;
  T mu4;                 // 4 / mu
  int sp;                // 1, 2, 0 = infinity
  int* err;              // set to 1 when a bounded wait gives up
  long long budget;      // clock cycles a bounded wait may take
  uint32_t probe;        // extra bytes armed on the first row's barrier (0; 16 in the wait test)
};

// Coefficients of u2 = V A for the prox of tau*||.||_{S_p} at V (R x 2) with Gram
// [[a, b], [b, c]] = V^T V. With V = U diag(s) W^T and shrunk values t, u2 = V W diag(g) W^T,
// g_i = t_i / s_i. Writing W diag(g) W^T = gbar I + kap [[hd, b], [b, -hd]], hd = (a - c)/2,
// kap = (g1 - g2) / (l1 - l2), the case formulas below have no cancellation at s1 = s2.
// The eigen-decomposition of the symmetric 2 x 2 Gram matrix is one Jacobi rotation; the
// closed form needs no rotation angle, and where both singular values are shrunk (or both
// kept) no division by the eigenvalue gap, so it stays accurate in FP32 when the two values
// coincide. Where exactly one is shrunk, kap = g1 / (2 r) is a bounded ratio whose two factors
// vanish together (g1 <= (s1 - s2) / s1).
template <typename T>
__device__ __forceinline__ void schatten_coeffs(T a, T b, T c, T tau, int sp, T& A11, T& A12,
                                                T& A22) {
  const T tr = a + c;
  T gbar = T(0), kap = T(0);
  const T hd = T(0.5) * (a - c);
  if (sp == 2) {
    const T nf = sqrt(tr);
    gbar = (nf > tau) ? T(1) - tau / nf : T(0);
  } else if (tr > T(0)) {
    const T r = sqrt(hd * hd + b * b);             // (l1 - l2) / 2
    const T l1 = T(0.5) * tr + r;
    const T l2 = fmax(T(0.5) * tr - r, T(0));
    const T s1 = sqrt(l1), s2 = sqrt(l2);
    if (sp == 1) {
      if (s1 > tau) {
        if (s2 > tau) {
          const T q = s1 * s2;
          gbar = T(1) - tau * (s1 + s2) / (T(2) * q);
          kap = tau / (q * (s1 + s2));
        } else {
          const T g1 = T(1) - tau / s1;
          gbar = T(0.5) * g1;
          kap = (r > T(0)) ? g1 / (T(2) * r) : T(0);
        }
      }
    } else {  // p = infinity: t = s - proj_{tau B1}(s)
      if (s1 + s2 > tau) {
        if (s1 - s2 >= tau) {
          const T g1 = T(1) - tau / s1;  // g2 = 1
          gbar = T(0.5) * (g1 + T(1));
          kap = (r > T(0)) ? (g1 - T(1)) / (T(2) * r) : T(0);
        } else {
          const T t = T(0.5) * (s1 + s2 - tau);  // both shrink to t; here s2 > 0
          const T q = s1 * s2;
          gbar = t * (s1 + s2) / (T(2) * q);
          kap = -t / (q * (s1 + s2));
        }
      }
    }
  } else if (!(tau > T(0))) {
    gbar = T(1);
  }
  A11 = gbar + kap * hd;
  A22 = gbar - kap * hd;
  A12 = kap * b;
}

// Coefficients of the new dual d2' = u2 - V = V B, B = A - I of schatten_coeffs, from the Gram
// entries, and 1 / (mu s) of the data prox (s the positive root of s^2 - pv s - q / 4 = 0, q = 4 pp / mu)
// from pv = p^T v1 and pp = |p|^2. Q1, Q2 are the quotients the Schatten cases need, n / d each.
template <typename T>
struct SchCase {
  T n1, d1, n2, d2;      // gm = c0 + c1 n1 / d1,  kap = c2 n2 / d2
  T c0, c1, c2;
};
template <typename T>
__device__ __forceinline__ SchCase<T> schatten_case(T tr, T r, T s1, T s2, T tau, int sp) {
  // r: (l1 - l2) / 2 (p = 2: the Frobenius norm); s1 >= s2 the singular values
  SchCase<T> c{T(0), T(1), T(0), T(1), T(-1), T(0), T(0)};
  if (sp == 2) {
    if (r > tau) { c.n1 = tau; c.d1 = r; c.c0 = T(0); c.c1 = T(-1); }
  } else if (!(tr > T(0))) {
    if (!(tau > T(0))) c.c0 = T(0);
  } else if (sp == 1) {
    if (s2 > tau) {         // both shrink by tau
      const T q = s1 * s2, s = s1 + s2;
      c.n1 = tau * s; c.d1 = T(2) * q; c.c0 = T(0); c.c1 = T(-1);
      c.n2 = tau; c.d2 = q * s; c.c2 = T(1);
    } else if (s1 > tau) {  // 1 - tau / s1 and 0
      c.n1 = tau; c.d1 = s1; c.c0 = c.c1 = T(-0.5);
      if (r > T(0)) { c.n2 = s1 - tau; c.d2 = T(2) * r * s1; c.c2 = T(1); }
    }
  } else if (s1 + s2 > tau) {
    if (s1 - s2 >= tau) {   // 1 - tau / s1 and 1
      c.n1 = tau; c.d1 = s1; c.c0 = T(0); c.c1 = T(-0.5);
      if (r > T(0)) { c.n2 = tau; c.d2 = T(2) * r * s1; c.c2 = T(-1); }
    } else {                // both shrink to t = (s1 + s2 - tau) / 2; here s2 > 0
      const T q = s1 * s2, s = s1 + s2, t = T(0.5) * (s - tau);
      c.n1 = t * s; c.d1 = T(2) * q; c.c1 = T(1);
      c.n2 = t; c.d2 = q * s; c.c2 = T(-1);
    }
  }
  return c;
}
// Every lane of a group of G holds the same arguments and gets the same results. FP64 square
// roots and quotients cost a dozen operations each on a pipe of two lanes a clock: there the
// lanes of a group share them out, one instruction sequence for two roots or three quotients.
template <typename T, int G>
__device__ __forceinline__ void pixel_scalars(T a, T b, T c, T tau, int sp, T pv, T pp, T mu, T mu4,
                                              T& B11, T& B12, T& B22, T& c1n) {
  const T tr = a + c, hd = T(0.5) * (a - c), half = T(0.5) * tr;
  const T x = sp == 2 ? tr : hd * hd + b * b, y = pv * pv + mu4 * pp;
  T gm, kap;
  if constexpr (sizeof(T) == 8) {
    const int g = threadIdx.x & (G - 1);
    const T ra = sqrt((g & 1) ? y : x);
    const T r = __shfl_sync(0xffffffffu, ra, 0, G), disc = __shfl_sync(0xffffffffu, ra, 1, G);
    const T rb = sqrt((g & 1) ? fmax(half - r, T(0)) : half + r);
    const T s1 = __shfl_sync(0xffffffffu, rb, 0, G), s2 = __shfl_sync(0xffffffffu, rb, 1, G);
    const SchCase<T> k = schatten_case<T>(tr, r, s1, s2, tau, sp);
    const T n3 = pv >= T(0) ? T(2) : T(2) * (disc - pv), d3 = pv >= T(0) ? mu * (pv + disc) : T(4) * pp;
    const int l = g & 3;
    const T q = (l == 0 ? k.n1 : l == 1 ? k.n2 : n3) / (l == 0 ? k.d1 : l == 1 ? k.d2 : d3);
    gm = k.c0 + k.c1 * __shfl_sync(0xffffffffu, q, 0, G);
    kap = k.c2 * __shfl_sync(0xffffffffu, q, 1, G);
    c1n = __shfl_sync(0xffffffffu, q, 2, G);
  } else {
    const T disc = sqrt(y);
    // pv >= 0: 2 / (mu (pv + disc)); else the same root without cancellation, 4 pp = mu q
    c1n = pv >= T(0) ? T(2) / (mu * (pv + disc)) : T(2) * (disc - pv) / (T(4) * pp);
    const T r = sqrt(x);
    const T s1 = sqrt(half + r), s2 = sqrt(fmax(half - r, T(0)));
    const SchCase<T> k = schatten_case<T>(tr, r, s1, s2, tau, sp);
    gm = k.c0;
    kap = T(0);
    if (k.c1 != T(0)) gm += k.c1 * (k.n1 / k.d1);   // no quotient where everything shrinks to 0
    if (k.c2 != T(0)) kap = k.c2 * (k.n2 / k.d2);
  }
  B11 = gm + kap * hd;
  B22 = gm - kap * hd;
  B12 = kap * b;
}

template <typename T> struct Vec2Of;
template <> struct Vec2Of<float> { using type = float2; };
template <> struct Vec2Of<double> { using type = double2; };

// A second read of a staged pair, as its own load (the traced sweep needs the old d2 twice and has no
// registers to keep it).
__device__ __forceinline__ float2 ld_shared_again(const float2* p) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(smem_addr(p)));
  return v;
}
__device__ __forceinline__ double2 ld_shared_again(const double2* p) {
  double2 v;
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(smem_addr(p)));
  return v;
}

// Byte sizes of one pipeline stage (one tile row of d2, dloc and p, each with 16 bytes of
// alignment slack at both ends), for tiles at most NC pixels wide.
__host__ __device__ inline size_t al16(size_t v) { return (v + 15) / 16 * 16; }
// dls: local-dual values per pixel (K + 2 in the compact form, 3K in the full one).
template <typename T>
__host__ __device__ inline void stage_sizes(int NC, int L, int K, int dls, size_t& d2b, size_t& dlb,
                                            size_t& pb) {
  d2b = al16((size_t)NC * 2 * L * K * sizeof(T) + 32);
  dlb = al16((size_t)NC * dls * sizeof(T) + 32);
  pb = al16((size_t)NC * K * sizeof(T) + 32);
}

// Issue the bulk copies of one tile row (pixels [pix0, pix0 + TW)) into a stage.
// Each region starts at the 16-byte boundary at or below its first byte; returns nothing,
// the consumer recomputes the same offsets.
template <typename T>
__device__ __forceinline__ void issue_row(const SweepArgs<T>& a, size_t pix0, int TW, int L,
                                          unsigned char* st, int d2b, int dlb,
                                          uint64_t* bar, uint32_t extra = 0) {
  const int K = a.K;
  const int dls = a.cin ? K + 2 : 3 * K;   // local-dual values per pixel in the input form
  const char* g0 = reinterpret_cast<const char*>(a.d2) + pix0 * (2 * L * K * sizeof(T));
  const char* g1 = reinterpret_cast<const char*>(a.cin ? a.dcmp : a.dloc) + pix0 * (dls * sizeof(T));
  const char* g2 = reinterpret_cast<const char*>(a.p) + pix0 * (K * sizeof(T));
  const size_t n0 = (size_t)TW * 2 * L * K * sizeof(T);
  const size_t n1 = (size_t)TW * dls * sizeof(T);
  const size_t n2 = (size_t)TW * K * sizeof(T);
  const char* a0 = reinterpret_cast<const char*>(reinterpret_cast<uintptr_t>(g0) & ~uintptr_t(15));
  const char* a1 = reinterpret_cast<const char*>(reinterpret_cast<uintptr_t>(g1) & ~uintptr_t(15));
  const char* a2 = reinterpret_cast<const char*>(reinterpret_cast<uintptr_t>(g2) & ~uintptr_t(15));
  const uint32_t b0 = (uint32_t)al16((g0 - a0) + n0);
  const uint32_t b1 = (uint32_t)al16((g1 - a1) + n1);
  const uint32_t b2 = (uint32_t)al16((g2 - a2) + n2);
  mbar_arrive_expect_tx(bar, b0 + b1 + b2 + extra);
  bulk_g2s(st, a0, b0, bar);
  bulk_g2s(st + d2b, a1, b1, bar);
  bulk_g2s(st + d2b + dlb, a2, b2, bar);
}

// Deterministic flush of one window row: every thread column c writes its E contributions
// to exclusive slots (columns c .. c+E-1 of the tile+halo row), the block synchronises, and
// the owner of each (column, class) sums the E slots in order s = 0..E-1 and stores the result
// straight into row `ey` of the tile's partials (each tile+halo row is flushed exactly once).
// Slots of idle columns stay zero. po: offset of the thread's class in the tile's partials.
template <typename T, int G, int NT, int E, bool DIAG>
__device__ __forceinline__ void flush_write(const T (&w)[E], const T (&w2)[DIAG ? E : 1], bool colok,
                                            int c, int g, T* slots, T* slots2) {
  constexpr int SW = NT / G + E - 1;
  if (colok) {
#pragma unroll
    for (int s = 0; s < E; ++s) {
      slots[(s * SW + c + s) * G + g] = w[s];
      if constexpr (DIAG) slots2[(s * SW + c + s) * G + g] = w2[s];
    }
  }
}
template <typename T, int G, int NT, int E, bool DIAG>
__device__ __forceinline__ void flush_sum(int c, int g, const T* slots, const T* slots2, T* Pt, T* Pt2,
                                          int ey, int EWmax, int EW, int K, int pstr, int po) {
  constexpr int NCT = NT / G;
  constexpr int SW = NCT + E - 1;
  if (g >= K) return;
  const int q = ey * EWmax;
#pragma unroll
  for (int r = 0; r < (SW + NCT - 1) / NCT; ++r) {
    const int col = c + r * NCT;
    if (col < EW) {
      T sum = T(0), sum2 = T(0);
#pragma unroll
      for (int s = 0; s < E; ++s) {
        sum += slots[(s * SW + col) * G + g];
        if constexpr (DIAG) sum2 += slots2[(s * SW + col) * G + g];
      }
      Pt[(q + col) * pstr + po] = sum;
      if constexpr (DIAG) Pt2[(q + col) * K + g] = sum2;
    }
  }
}

// Warps an SM holds: 24 for the FP32 variants up to 3 x 3 (80 registers), 16 otherwise. The traced
// ones take 80 registers only with compile-time class strides (2048 x 2048, K = 16: a trace costs 846 us
// with 16 warps, 735 with 24; 400 x 300, K = 9: 55 against 69, its spills outweigh them).
template <typename T, int M, bool DIAG, bool KEQ, int NT>
constexpr int sweep_min_blocks() {
  return ((sizeof(T) == 8 || M >= 2 || (DIAG && !KEQ)) ? 2 : 3) * (256 / NT);
}

// Flush slot buffers: two in FP32, so that one barrier a row orders them (and the stages); FP64 and
// the simplex and traced forms, whose stages or slots are larger, keep one and a second barrier.
template <typename T, bool DIAG, bool SIMP>
constexpr int sweep_slot_bufs() { return (sizeof(T) == 4 && !SIMP && !DIAG) ? 2 : 1; }

// SIMP selects the MPO of g4: false, the projection onto the affine set 1^T xi = 1 (eq. 10);
// true, the projection onto the probability simplex (Sec. 4's description of that MPO).
// KEQ: the class count equals the lane count G, so the class strides are compile-time constants
// (measured 8 % fewer sweep cycles at 145 x 145, K = 16). NT: threads of a CTA.
template <typename T, int M, int G, bool DIAG, bool SIMP, bool KEQ, int NT>
__global__ void __launch_bounds__(NT, sweep_min_blocks<T, M, DIAG, KEQ, NT>()) k_sweep(const SweepArgs<T> a) {
  constexpr int L = (2 * M + 1) * (2 * M + 1);
  constexpr int E = 2 * M + 2;
  constexpr int SB = sweep_slot_bufs<T, DIAG, SIMP>();
  using V2 = typename Vec2Of<T>::type;

  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* mbar = reinterpret_cast<uint64_t*>(smem_raw);  // 2 stage barriers
  const GiveUp gave_up{reinterpret_cast<int*>(smem_raw + 32)};
  const int K = KEQ ? G : a.K;
  const bool cin = !SIMP && a.cin;      // the simplex sweep always reads the full form
  const int dls = cin ? K + 2 : 3 * K;
  size_t d2b_, dlb_, pb_;
  stage_sizes<T>(KEQ ? NT / G : a.NC, L, K, dls, d2b_, dlb_, pb_);
  const int d2b = (int)d2b_, dlb = (int)dlb_, stb = d2b + dlb + (int)pb_;
  unsigned char* stage0 = smem_raw + 128;
  const int slot = a.EHmax * a.EWmax * G;
  T* zs = reinterpret_cast<T*>(stage0 + 2 * stb);
  T* om = zs + slot;                    // [L]
  // flush slots: row contributions of thread column c for tile+halo column c + s live at
  // slots[(s * SW + c + s) * G + g]; each (s, column) has one writer, owners sum over s
  constexpr int SW = NT / G + E - 1;    // columns of a slot row (NC <= NT / G)
  constexpr int SLOTS = E * SW * G;
  T* slots = om + ((L + 3) & ~3);       // [SB][DIAG ? 2 : 1][SLOTS]
  constexpr int SBUF = (DIAG ? 2 : 1) * SLOTS;
  __shared__ double red32[32];

  const int tile = blockIdx.x;
  const int ty = tile / a.ntx, tx = tile - ty * a.ntx;
  const int y0 = (int)(((long long)ty * a.H) / a.nty);
  const int y1 = (int)(((long long)(ty + 1) * a.H) / a.nty);
  const int x0 = (int)(((long long)tx * a.W) / a.ntx);
  const int x1 = (int)(((long long)(tx + 1) * a.W) / a.ntx);
  const int TH = y1 - y0, TW = x1 - x0;
  const int EH = TH + 2 * M + 1, EW = TW + 2 * M + 1;
  const int g = threadIdx.x % G, c = threadIdx.x / G;
  // this tile's partials (tile + halo)
  T* Pt = a.P + (size_t)tile * a.ptile;
  T* Pt2 = DIAG ? a.P2 + (size_t)tile * a.EHmax * a.EWmax * K : nullptr;
  const int po = (g >> 2) * a.pquad + (g & 3);

  if (threadIdx.x == 0) {
    mbar_init(&mbar[0], 1);
    mbar_init(&mbar[1], 1);
    mbar_fence_init();
    gave_up.clear();
  }
  for (int j = threadIdx.x; j < L; j += NT) om[j] = a.omega[j];
  for (int j = threadIdx.x; j < SB * SBUF; j += NT) slots[j] = T(0);
  pdl_wait();  // z, d, p and the partial buffers belong to the previous kernels
  __syncthreads();
  if (threadIdx.x == 0) {
    issue_row<T>(a, (size_t)y0 * a.W + x0, TW, L, stage0, d2b, dlb, &mbar[0], a.probe);
    if (TH > 1) issue_row<T>(a, (size_t)(y0 + 1) * a.W + x0, TW, L, stage0 + stb, d2b, dlb, &mbar[1]);
  }
  // z tile (with halo, periodic) by per-thread async copies of 16 bytes where a pixel's classes are
  // whole vectors, else value by value; padded classes read as zero. Threads stride by whole
  // pixels, so (ex, ey) advance incrementally (no runtime division in the loop)
  {
    constexpr int VE = 16 / sizeof(T);
    const bool vec = KEQ || K % VE == 0;
    const int per = vec ? G / VE : G;             // copies of a pixel
    const int PS = NT / per;
    const int k = (threadIdx.x & (per - 1)) * (vec ? VE : 1);
    const int p0 = threadIdx.x / per;
    int ex = p0 % a.EWmax, ey = p0 / a.EWmax;
    while (ey < EH) {
      const bool v = k < K && ex < EW;
      const T* src = a.z;
      if (v) {
        int y = y0 - M + ey, xx = x0 - M + ex;
        y += (y < 0) ? a.H : 0;
        y -= (y >= a.H) ? a.H : 0;
        xx += (xx < 0) ? a.W : 0;
        xx -= (xx >= a.W) ? a.W : 0;
        src = a.z + ((size_t)y * a.W + xx) * K + k;
      }
      T* dst = zs + (ey * a.EWmax + ex) * G + k;
      if (vec) cp_async_zfill<16>(dst, src, v);
      else cp_async_zfill<sizeof(T)>(dst, src, v);
      ex += PS;
      while (ex >= a.EWmax) { ex -= a.EWmax; ++ey; }
    }
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();

  const bool colok = c < TW;
  const bool kok = colok && (KEQ || g < K);
  const int cc = colok ? c : 0;                   // idle columns read column 0
  // KEQ instantiations run only with full-width tiles (NC = NT / G), so their z-tile row
  // stride is a compile-time constant too
  const int EWs = KEQ ? NT / G + 2 * M + 1 : a.EWmax;

  T accW[E][E];
  constexpr int E2 = DIAG ? E : 1;
  T accW2[E2][E2];
#pragma unroll
  for (int r = 0; r < E; ++r)
#pragma unroll
    for (int s = 0; s < E; ++s) accW[r][s] = T(0);
#pragma unroll
  for (int r = 0; r < E2; ++r)
#pragma unroll
    for (int s = 0; s < E2; ++s) accW2[r][s] = T(0);
  T sq = T(0);
  const T tau = a.tau;
  // shift weights in registers for the FP32 3 x 3 patch (the 5 x 5 and FP64 variants are at
  // their register caps)
  constexpr bool OMR = M <= 1 && sizeof(T) == 4;
  constexpr int LR = OMR ? L : 1;
  T omr[LR];
#pragma unroll
  for (int j = 0; j < LR; ++j) omr[j] = om[j];
  auto omega_j = [&](int j) -> T { return OMR ? omr[j < LR ? j : 0] : om[j]; };
  // the staged regions start at the 16-byte boundary at or below a row's first value (as
  // issue_row): the offsets of the three, from the low address bits alone
  const uint32_t l0 = (uint32_t)reinterpret_cast<uintptr_t>(a.d2);
  const uint32_t l1 = (uint32_t)reinterpret_cast<uintptr_t>(cin ? a.dcmp : a.dloc);
  const uint32_t l2 = (uint32_t)reinterpret_cast<uintptr_t>(a.p);

  for (int r = 0; r < TH; ++r) {
    const int sidx = r & 1;
    if constexpr (SB == 1) __syncthreads();       // the slots' owners are done with them
    if (!mbar_wait_bounded(&mbar[sidx], (uint32_t)((r >> 1) & 1), a.budget)) gave_up.raise(r);
    const size_t pix0 = (size_t)(y0 + r) * a.W + x0;  // the row's first pixel
    const uint32_t pl = (uint32_t)pix0;               // (its low bits suffice for the offsets)
    unsigned char* st = stage0 + sidx * stb;
    const uint32_t f0 = (l0 + pl * (uint32_t)(2 * L * K * sizeof(T))) & 15;
    const uint32_t f1 = (l1 + pl * (uint32_t)(dls * sizeof(T))) & 15;
    const uint32_t f2 = (l2 + pl * (uint32_t)(K * sizeof(T))) & 15;
    const V2* sd2 = reinterpret_cast<const V2*>(st + f0) + cc * L * K + g;
    const T* sdp = reinterpret_cast<const T*>(st + d2b + f1) + cc * dls;  // pixel
    const T* sp = reinterpret_cast<const T*>(st + d2b + dlb + f2) + cc * K + g;
    // ---- loads: duals and p of this pixel / class (from the staged row). Idle columns compute
    // what reaches no other column's sums, slots or stores; idle lanes of a live pixel (g >= K
    // read the next values of the stage) are masked where they would reach the group sums
    V2 dv[L];
#pragma unroll
    for (int j = 0; j < L; ++j) dv[j] = sd2[j * K];
    T pk = sp[0], d1, d3, d4;
    if (cin) {              // d1 = c1 p, d4 = c4 1 (the forms the MPOs of g1 and g4 leave)
      d3 = sdp[g];
      d1 = sdp[K] * pk;
      d4 = sdp[K + 1];
    } else {
      d1 = sdp[g];
      d3 = sdp[K + g];
      d4 = sdp[2 * K + g];
    }
    // ---- v2 = J z - d2 (eq. 4), from the shared tile, and the Gram matrix (eq. 5) over the (j, k)
    // rows of this pixel
    const T* zc = zs + ((r + M) * EWs + (cc + M)) * G + g;
    T vh[L], vv[L];
    T ga = T(0), gb = T(0), gc = T(0);
    T zt[E], zb[E];                               // z of the window's rows dy and dy + 1
#pragma unroll
    for (int s = 0; s < E; ++s) zt[s] = zc[(-M * EWs + s - M) * G];
#pragma unroll
    for (int dy = -M; dy <= M; ++dy) {
#pragma unroll
      for (int s = 0; s < E; ++s) zb[s] = zc[((dy + 1) * EWs + s - M) * G];
#pragma unroll
      for (int dx = -M; dx <= M; ++dx) {
        const int j = (dy + M) * (2 * M + 1) + (dx + M);
        const T w = omega_j(j);
        vh[j] = w * (zt[dx + M + 1] - zt[dx + M]) - dv[j].x;
        vv[j] = w * (zb[dx + M] - zt[dx + M]) - dv[j].y;
        ga += vh[j] * vh[j];
        gb += vh[j] * vv[j];
        gc += vv[j] * vv[j];
      }
#pragma unroll
      for (int s = 0; s < E; ++s) zt[s] = zb[s];
    }
    const T z0 = zc[0];
    const T v1 = z0 - d1, v3 = z0 - d3, v4 = z0 - d4;
    T pv = pk * v1, pp = pk * pk, s4 = v4;
    if constexpr (!KEQ) {
      if (g >= K) { ga = gb = gc = T(0); pv = pp = s4 = T(0); }
    }
    ga = group_sum<G>(ga);
    gb = group_sum<G>(gb);
    gc = group_sum<G>(gc);
    pv = group_sum<G>(pv);
    pp = group_sum<G>(pp);
    if constexpr (!SIMP) s4 = group_sum<G>(s4);
    T B11, B12, B22, c1n;
    pixel_scalars<T, G>(ga, gb, gc, tau, a.sp, pv, pp, a.mu, a.mu4, B11, B12, B22, c1n);
    // ---- pixel-local MPOs of g1, g3, g4 and their duals. The new d1 is p / (mu s) = c1 p and, for
    // the affine g4, the new d4 is the same -(1^T v4 - 1) / K for every class: the compact form
    // stores c1 and c4 per pixel
    const T n1 = pk * c1n, u1 = v1 + n1;
    const T u3 = fmax(v3, T(0)), n3 = u3 - v3;
    T u4, n4;
    if constexpr (!SIMP) {
      n4 = -(s4 - T(1)) * a.invK;
      u4 = v4 + n4;
    } else {
      // Michelot: threshold over the active classes until no class leaves the active set (at
      // most K passes; the loop runs until no group of the warp changes, so that every lane
      // takes part in the shuffles)
      bool act = kok;
      T theta = T(0);
      for (int pass = 0; pass < 32; ++pass) {
        const T cnt = group_sum<G>(act ? T(1) : T(0));
        const T sum = group_sum<G>(act ? v4 : T(0));
        theta = (cnt > T(0)) ? (sum - T(1)) / cnt : T(0);
        const bool nact = act && (v4 > theta);
        const bool changed = nact != act;
        act = nact;
        if (!__any_sync(0xffffffffu, changed)) break;
      }
      u4 = kok ? fmax(v4 - theta, T(0)) : T(0);
      n4 = u4 - v4;
    }
    if constexpr (SIMP) {
      if (kok) {
        T* dl = a.dloco + pix0 * 3 * K + (cc * 3 * K + g);
        dl[0] = n1;
        dl[K] = n3;
        dl[2 * K] = n4;
      }
    } else {
      T* dc = a.dcmp + pix0 * (K + 2) + cc * (K + 2);
      if (kok) dc[g] = n3;
      if (kok && g == 0) {
        dc[K] = c1n;
        dc[K + 1] = n4;
      }
    }
    accW[M][M] += (u1 + n1) + (u3 + n3) + (u4 + n4);
    if constexpr (DIAG) {
      accW2[M][M] += n1 + n3 + n4;
      if (kok) sq += (n1 - d1) * (n1 - d1) + (n3 - d3) * (n3 - d3) + (n4 - d4) * (n4 - d4);
    }
    // ---- the new d2 = V B, w = u2 + d2 = V + 2 d2 and its J^T scatter into the window
#pragma unroll
    for (int s = 0; s < E; ++s) {                 // the window's new bottom row
      accW[E - 1][s] = T(0);
      if constexpr (DIAG) accW2[E - 1][s] = T(0);
    }
    V2* d2w = reinterpret_cast<V2*>(a.d2o) + pix0 * L * K + (cc * L * K + g);
#pragma unroll
    for (int dy = -M; dy <= M; ++dy)
#pragma unroll
      for (int dx = -M; dx <= M; ++dx) {
        const int j = (dy + M) * (2 * M + 1) + (dx + M);
        const T nh = vh[j] * B11 + vv[j] * B12, nv = vh[j] * B12 + vv[j] * B22;
        if constexpr (DIAG) {
          const V2 od = ld_shared_again(sd2 + j * K);
          const T eh = nh - od.x, ev = nv - od.y;
          if (kok) sq += eh * eh + ev * ev;
        }
        if (kok) {
          V2 o; o.x = nh; o.y = nv;
          d2w[(size_t)j * K] = o;
        }
        const T w = omega_j(j);
        const T th = T(2) * nh + vh[j], tv = T(2) * nv + vv[j];
        accW[dy + M][dx + M + 1] += w * th;
        accW[dy + M][dx + M] -= w * (th + tv);
        accW[dy + M + 1][dx + M] += w * tv;
        if constexpr (DIAG) {
          accW2[dy + M][dx + M + 1] += w * nh;
          accW2[dy + M][dx + M] -= w * (nh + nv);
          accW2[dy + M + 1][dx + M] += w * nv;
        }
      }
    // ---- flush the finished top window row (tile+halo row r), in a fixed summation order
    T* sl = slots + (SB == 2 ? sidx * SBUF : 0);
    flush_write<T, G, NT, E, DIAG>(accW[0], accW2[0], colok, c, g, sl, sl + SLOTS);
    __syncthreads();       // slots written; every thread is past its reads of this row's stage
    if (gave_up.raised(r)) {   // uniform (giveup.h)
      // a copy never completed: report, give the copies in flight a bounded chance, and leave
      if (threadIdx.x == 0) {
        atomicExch(a.err, 1);
        mbar_wait_bounded(&mbar[sidx], (uint32_t)((r >> 1) & 1), drain_cycles(a.budget));
        if (r + 1 < TH)
          mbar_wait_bounded(&mbar[sidx ^ 1], (uint32_t)(((r + 1) >> 1) & 1), drain_cycles(a.budget));
      }
      return;
    }
    if (threadIdx.x == 0 && r + 2 < TH)
      issue_row<T>(a, (size_t)(y0 + r + 2) * a.W + x0, TW, L, st, d2b, dlb, &mbar[sidx]);
    flush_sum<T, G, NT, E, DIAG>(c, g, sl, sl + SLOTS, Pt, Pt2, r, EWs, EW, K, a.pstr, po);
#pragma unroll
    for (int rr = 0; rr < E - 1; ++rr)
#pragma unroll
      for (int s = 0; s < E; ++s) accW[rr][s] = accW[rr + 1][s];
    if constexpr (DIAG) {
#pragma unroll
      for (int rr = 0; rr < E - 1; ++rr)
#pragma unroll
        for (int s = 0; s < E; ++s) accW2[rr][s] = accW2[rr + 1][s];
    }
  }
  // remaining window rows: tile+halo rows TH .. TH + 2M
  pdl_trigger();
#pragma unroll
  for (int rr = 0; rr < E - 1; ++rr) {
    if constexpr (SB == 1) __syncthreads();  // the previous flush's owners are done with the slots
    T* sl = slots + (SB == 2 ? ((TH + rr) & 1) * SBUF : 0);
    flush_write<T, G, NT, E, DIAG>(accW[rr], accW2[DIAG ? rr : 0], colok, c, g, sl, sl + SLOTS);
    __syncthreads();
    flush_sum<T, G, NT, E, DIAG>(c, g, sl, sl + SLOTS, Pt, Pt2, TH + rr, EWs, EW, K, a.pstr, po);
  }
  if constexpr (DIAG) {
    const double t = block_sum_w<T>(sq, red32);
    if (threadIdx.x == 0) a.diag_sq[tile] = t;
  }
}

// Largest dynamic shared memory granted so far to each sweep variant.
template <typename T, int M, int G, bool DIAG, bool SIMP, bool KEQ, int NT>
struct SweepGrant {
  static SmemGrants v;
};
template <typename T, int M, int G, bool DIAG, bool SIMP, bool KEQ, int NT>
SmemGrants SweepGrant<T, M, G, DIAG, SIMP, KEQ, NT>::v;

// Shared memory of one sweep CTA of nt threads in bytes: barriers, two row stages, z tile, flush
// slots. compact: the local duals come in compact form.
template <typename T>
inline size_t sweep_smem_bytes(int nt, int NC, int EHmax, int EWmax, int G, int L, int K, bool diag,
                               bool compact, bool simplex) {
  size_t d2b, dlb, pb;
  stage_sizes<T>(NC, L, K, compact ? K + 2 : 3 * K, d2b, dlb, pb);
  const int E = EWmax - NC;  // 2M + 1 ... the window width is E + 1 = 2M + 2
  const size_t slots = (size_t)(E + 1) * (nt / G + E) * G * (sizeof(T) == 4 && !simplex && !diag ? 2 : 1);
  return 128 + 2 * (d2b + dlb + pb) +
         sizeof(T) * ((size_t)EHmax * EWmax * G + (size_t)((L + 3) & ~3) +
                      (diag ? 2 : 1) * slots);
}

// grid = 0: only grant the shared memory (so that graph capture never changes attributes).
template <typename T, int M, int G, bool DIAG, bool SIMP, bool KEQ, int NT>
inline cudaError_t launch_sweep_inst(const SweepArgs<T>& a, int tiles, size_t smem, cudaStream_t st) {
  cudaError_t e = grant_smem(k_sweep<T, M, G, DIAG, SIMP, KEQ, NT>, smem,
                             SweepGrant<T, M, G, DIAG, SIMP, KEQ, NT>::v);
  if (e != cudaSuccess || tiles == 0) return e;
  return launch_pdl_carve(true, k_sweep<T, M, G, DIAG, SIMP, KEQ, NT>, dim3(tiles), dim3(NT), smem, st, a);
}

// CTAs of 64 threads where their 64 / G columns still are a tile (at least 2M + 1).
constexpr bool sweep_small_ok(int M, int G) { return 64 / G >= 2 * M + 1; }

template <typename T, int M, int G, bool DIAG, bool SIMP, bool KEQ>
inline cudaError_t launch_sweep_nt(const SweepArgs<T>& a, int nt, int tiles, size_t smem, cudaStream_t st) {
  if constexpr (sweep_small_ok(M, G))
    if (nt == 64) return launch_sweep_inst<T, M, G, DIAG, SIMP, KEQ, 64>(a, tiles, smem, st);
  return launch_sweep_inst<T, M, G, DIAG, SIMP, KEQ, 256>(a, tiles, smem, st);
}

template <typename T, int M, bool DIAG, bool SIMP, bool KEQ>
inline cudaError_t launch_sweep_g(const SweepArgs<T>& a, int G, int nt, int tiles, size_t smem,
                                  cudaStream_t st) {
  switch (G) {
    case 4: return launch_sweep_nt<T, M, 4, DIAG, SIMP, KEQ>(a, nt, tiles, smem, st);
    case 8: return launch_sweep_nt<T, M, 8, DIAG, SIMP, KEQ>(a, nt, tiles, smem, st);
    case 16: return launch_sweep_nt<T, M, 16, DIAG, SIMP, KEQ>(a, nt, tiles, smem, st);
    case 32: return launch_sweep_nt<T, M, 32, DIAG, SIMP, KEQ>(a, nt, tiles, smem, st);
  }
  return cudaErrorInvalidValue;
}

template <typename T, bool DIAG, bool SIMP, bool KEQ>
inline cudaError_t launch_sweep_md(const SweepArgs<T>& a, int M, int G, int nt, int tiles, size_t smem,
                                   cudaStream_t st) {
  switch (M) {
    case 0: return launch_sweep_g<T, 0, DIAG, SIMP, KEQ>(a, G, nt, tiles, smem, st);
    case 1: return launch_sweep_g<T, 1, DIAG, SIMP, KEQ>(a, G, nt, tiles, smem, st);
    case 2: return launch_sweep_g<T, 2, DIAG, SIMP, KEQ>(a, G, nt, tiles, smem, st);
  }
  return cudaErrorInvalidValue;
}

// The instantiations of one precision and one g4 variant (each in its own translation unit).
template <typename T, bool SIMP, bool KEQ>
inline cudaError_t launch_sweep_variant(const SweepArgs<T>& a, int M, int G, int nt, bool diag,
                                        int tiles, size_t smem, cudaStream_t st) {
  return diag ? launch_sweep_md<T, true, SIMP, KEQ>(a, M, G, nt, tiles, smem, st)
              : launch_sweep_md<T, false, SIMP, KEQ>(a, M, G, nt, tiles, smem, st);
}

}  // namespace sgs
