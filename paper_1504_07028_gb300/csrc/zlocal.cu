// Kernel and launcher of the pixel-domain z-update (zlocal.cuh has the method).
#include "zlocal.cuh"

namespace sgs {

// Two FP32 values in one 64-bit register pair: one instruction for two points.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pk2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f32x2 pk2(float2 v) { return pk2(v.x, v.y); }
__device__ __forceinline__ float lo2(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a;
}
__device__ __forceinline__ float hi2(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return b;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ void acc4(float4& v, const float4 w) {
  v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
}

// ------------------------------------------------------------ streaming form (large images)
//
// A CTA takes a strip of ZL_WIDTH columns of one class quad, a warp each class; a lane holds four
// adjacent columns. The rows of the strip stream through a window of WIN rows in registers (per
// row the even and the odd columns as pairs): row r enters at time r with step 1 and gets step
// k at time r + k - 1, so at time t step k works on row t - k + 1, from the newest row to the
// oldest; a row's right-hand neighbour below has had step k - 1 by then, its neighbour above
// too, and it leaves after step 17. All steps of one time update the columns of one parity, and the only
// value from another lane is one edge column of each row (a shuffle). No halo rows are computed
// twice within a segment, no barrier orders the steps; one barrier a row hands over the staged
// input row (px-major loads of four classes, transposed through shared memory) and the
// finished row.
constexpr int ZS_WIN = ZL_STEPS + 1;


// Rows in flight: every thread copies its own column of a row (four classes, up to 2 x 2 covers)
// into the row's slot ZS_DEPTH rows ahead, and reads it back itself, so a row's arrival needs
// no barrier.
constexpr int ZS_DEPTH = 6;               // also the rows of one unrolled block (an even number)
template <int MODE>
constexpr int zs_covers() { return MODE == 0 ? 4 : 1; }
template <int MODE>
constexpr size_t zs_smem() { return sizeof(float4) * ZS_DEPTH * zs_covers<MODE>() * ZL_WIDTH; }

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// MODE: 0 tile partials, 1 dense rhs in 16-byte vectors, 2 dense rhs value by value. Starts the
// copies of one row: src points at this thread's pixel of a dense row; cy, ox0, ox1 give the
// covers of a row of partials.
template <int MODE>
__device__ __forceinline__ void zs_issue(const ZlArgs& a, float4* slot, const float* src, int nv, int ox0,
                                         int ox1, int2 cy) {
  if constexpr (MODE == 0) {
    const float4* P = reinterpret_cast<const float4*>(a.P);
    cp_async16(slot, P + (cy.x + ox0));
    if (ox1 >= 0) cp_async16(slot + ZL_WIDTH, P + (cy.x + ox1));
    if (cy.y >= 0) {
      cp_async16(slot + 2 * ZL_WIDTH, P + (cy.y + ox0));
      if (ox1 >= 0) cp_async16(slot + 3 * ZL_WIDTH, P + (cy.y + ox1));
    }
  } else if constexpr (MODE == 1) {
    cp_async16(slot, src);
  } else {
    float* d = reinterpret_cast<float*>(slot);
#pragma unroll
    for (int j = 0; j < 4; ++j) cp_async_zfill<4>(d + j, j < nv ? src + j : src, j < nv);
  }
}

template <int MODE, bool VEC>
__global__ void __launch_bounds__(128, 2) k_zstream(const ZlArgs a) {
  __shared__ __align__(16) float in[2][4][ZL_WIDTH], out[2][4][ZL_WIDTH];
  extern __shared__ __align__(128) unsigned char smem_raw[];
  constexpr int NCOV = zs_covers<MODE>();
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  float4* ring = reinterpret_cast<float4*>(smem_raw) + tid;   // [ZS_DEPTH][NCOV][ZL_WIDTH]
  int u = blockIdx.x;
  const int cg = u % a.ng;
  u /= a.ng;
  const int sx = u % a.p.nx, sy = u / a.p.nx;
  const int x0 = (int)(((long long)sx * a.W) / a.p.nx), x1 = (int)(((long long)(sx + 1) * a.W) / a.p.nx);
  const int y0 = (int)(((long long)sy * a.H) / a.p.ny), y1 = (int)(((long long)(sy + 1) * a.H) / a.p.ny);
  const int R = y1 - y0 + 2 * ZL_HALO;           // input rows y0 - ZL_HALO ..
  const int T = y1 - y0 + ZL_HALO + ZL_STEPS - 1;  // the last wanted row leaves at time T - 1
  const int x = x0 - ZL_HALO + tid;              // this thread's column of the staged rows
  const int gx = wrap_idx(x, a.W);
  const bool mine = x >= x0 && x < x1;
  const int nv = min(4, a.K - 4 * cg);           // classes of this quad
  int gy = wrap_idx(y0 - ZL_HALO, a.H);          // image row of the next copy
  int ox0 = 0, ox1 = -1;
  if constexpr (MODE == 0) {
    const int2 cx = __ldg(reinterpret_cast<const int2*>(a.covX) + gx);
    const int pl = a.EHmax * a.EWmax;
    ox0 = ((cx.x >> 16) * a.ng + cg) * pl + (cx.x & 0xffff);
    if (cx.y >= 0) ox1 = ((cx.y >> 16) * a.ng + cg) * pl + (cx.y & 0xffff);
  }
  const size_t rowK = (size_t)a.W * a.K;
  const float* src = MODE == 0 ? nullptr : a.src + (size_t)gx * a.K + 4 * cg;
  float* zp = a.z + ((size_t)y0 * a.W + (mine ? x : 0)) * a.K + 4 * cg;  // this thread's next output
  const f32x2 cw = pk2(a.q.cw[ZL_EARLY]), c1 = pk2(a.q.c1[ZL_EARLY]);
  // rows of the window: at the start of a block of ZS_DEPTH steps, entry i is row t0 - ZS_WIN + i;
  // the block's own rows take entries ZS_WIN ..
  f32x2 xE[ZS_WIN + ZS_DEPTH], xO[ZS_WIN + ZS_DEPTH], bE[ZS_WIN + ZS_DEPTH], bO[ZS_WIN + ZS_DEPTH];
#pragma unroll
  for (int i = 0; i < ZS_WIN + ZS_DEPTH; ++i) xE[i] = xO[i] = bE[i] = bO[i] = 0;
  // copies of row r into slot r mod ZS_DEPTH; the vertical covers are fetched one row ahead
  int2 cy = make_int2(0, -1);
  bool hy[ZS_DEPTH];                              // the slot's row has a second vertical cover
  if constexpr (MODE == 0) cy = __ldg(reinterpret_cast<const int2*>(a.offY) + gy);
  pdl_wait();  // the rhs comes from the previous kernel
  auto issue = [&](int slot, int r) {
    if (r < R) {
      zs_issue<MODE>(a, ring + slot * NCOV * ZL_WIDTH, MODE == 0 ? nullptr : src + gy * rowK, nv, ox0, ox1, cy);
      hy[slot] = cy.y >= 0;
      gy = gy + 1 == a.H ? 0 : gy + 1;
      if constexpr (MODE == 0) cy = __ldg(reinterpret_cast<const int2*>(a.offY) + gy);
    }
    cp_async_commit();
  };
  // row r of the slot, summed and transposed
  auto stage = [&](int buf, int slot, int r) {
    cp_async_wait_group<ZS_DEPTH - 1>();
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < R) {
      const float4* q = ring + slot * NCOV * ZL_WIDTH;
      v = q[0];
      if constexpr (MODE == 0) {
        if (ox1 >= 0) acc4(v, q[ZL_WIDTH]);
        if (hy[slot]) {
          acc4(v, q[2 * ZL_WIDTH]);
          if (ox1 >= 0) acc4(v, q[3 * ZL_WIDTH]);
        }
      }
    }
    in[buf][0][tid] = v.x;
    in[buf][1][tid] = v.y;
    in[buf][2][tid] = v.z;
    in[buf][3][tid] = v.w;
  };
#pragma unroll
  for (int r = 0; r < ZS_DEPTH; ++r) issue(r, r);
  stage(0, 0, 0);
  const bool live = 4 * cg + w < a.K;             // this warp's class exists
  const f32x2 bs = pk2(make_float2(a.q.bs, a.q.bs)), b0 = pk2(a.q.b0);
  __syncthreads();
  for (int t0 = 0; t0 < T; t0 += ZS_DEPTH) {
#pragma unroll
    for (int s = 0; s < ZS_DEPTH; ++s) {
      const int t = t0 + s;
      if (t >= T) break;                          // uniform over the CTA
      issue(s, t + ZS_DEPTH);
      stage((s + 1) & 1, (s + 1) % ZS_DEPTH, t + 1);
      if (live) {
      const float4 bv = *reinterpret_cast<const float4*>(&in[s & 1][w][4 * lane]);
      constexpr int N0 = ZS_WIN;                  // entry of row t0
      bE[N0 + s] = mul2(pk2(bv.x, bv.z), bs);
      bO[N0 + s] = mul2(pk2(bv.y, bv.w), bs);
      xE[N0 + s] = s % 2 == 0 ? mul2(bE[N0 + s], b0) : 0;
      xO[N0 + s] = s % 2 == 0 ? 0 : mul2(bO[N0 + s], b0);
      // x_i <- w (left + right + above) + c1 x_i + b for every row of the window, none waiting for
      // another (newest first: a row's neighbour above still holds its old value), ...
#pragma unroll
      for (int k = 2; k <= ZL_STEPS; ++k) {
        const int i = N0 + s - k + 1, up = i - 1;
        const int e = k - 2 < ZL_EARLY ? k - 2 : ZL_EARLY;
        const f32x2 wk = e < ZL_EARLY ? pk2(a.q.cw[e]) : cw, ck = e < ZL_EARLY ? pk2(a.q.c1[e]) : c1;
        if (s % 2 == 0) {
          const float ext = __shfl_up_sync(0xffffffffu, hi2(xO[i]), 1);
          const f32x2 bb = e < ZL_EARLY ? mul2(bE[i], pk2(a.q.cb[e < ZL_EARLY ? e : 0])) : bE[i];
          const float o0 = lo2(xO[i]), o1 = hi2(xO[i]);
          const f32x2 h = add2(pk2(ext + o0, o0 + o1), xE[up]);
          xE[i] = fma2(h, wk, fma2(xE[i], ck, bb));
        } else {
          const float ext = __shfl_down_sync(0xffffffffu, lo2(xE[i]), 1);
          const f32x2 bb = e < ZL_EARLY ? mul2(bO[i], pk2(a.q.cb[e < ZL_EARLY ? e : 0])) : bO[i];
          const float e0 = lo2(xE[i]), e1 = hi2(xE[i]);
          const f32x2 h = add2(pk2(e0 + e1, e1 + ext), xO[up]);
          xO[i] = fma2(h, wk, fma2(xO[i], ck, bb));
        }
      }
      // ... then the neighbour below, already updated: one multiply-add a row in sequence
#pragma unroll
      for (int k = 2; k <= ZL_STEPS; ++k) {
        const int i = N0 + s - k + 1, dn = i + 1;
        const int e = k - 2 < ZL_EARLY ? k - 2 : ZL_EARLY;
        const f32x2 wk = e < ZL_EARLY ? pk2(a.q.cw[e]) : cw;
        if (s % 2 == 0) xE[i] = fma2(xE[dn], wk, xE[i]);
        else xO[i] = fma2(xO[dn], wk, xO[i]);
      }
      const int f = N0 + s - ZL_STEPS + 1;   // the row that leaves
      *reinterpret_cast<float4*>(&out[s & 1][w][4 * lane]) =
          make_float4(lo2(xE[f]), lo2(xO[f]), hi2(xE[f]), hi2(xO[f]));
      }
      __syncthreads();
      if (t >= ZL_HALO + ZL_STEPS - 1) {          // rows y0 .. y1 - 1
        if (mine) {
          const float4 o = make_float4(out[s & 1][0][tid], out[s & 1][1][tid], out[s & 1][2][tid], out[s & 1][3][tid]);
          if constexpr (VEC) {
            *reinterpret_cast<float4*>(zp) = o;
          } else {
            zp[0] = o.x;
            if (nv > 1) zp[1] = o.y;
            if (nv > 2) zp[2] = o.z;
            if (nv > 3) zp[3] = o.w;
          }
        }
        zp += rowK;
      }
    }
#pragma unroll
    for (int i = 0; i < ZS_WIN; ++i) {
      xE[i] = xE[i + ZS_DEPTH]; xO[i] = xO[i + ZS_DEPTH];
      bE[i] = bE[i + ZS_DEPTH]; bO[i] = bO[i + ZS_DEPTH];
    }
  }
  pdl_trigger();
  cp_async_wait_all();                            // nothing may be in flight when the CTA exits
}

// ------------------------------------------------------------------ block form (small images)
//
// A thread holds a 4 x ZB_ROWS block of one class in registers, the even and the odd columns of a
// row as pairs; the threads of a CTA cover a tile with its halo for KC classes (class fastest).
// After a step every thread publishes the points it just updated on its block's edges; the
// next step, on the other colour, reads the four neighbours' edges: one barrier a step, 17
// short steps in all, where the streaming form takes a time step for every row. The halo costs
// this form several times the tile itself, so it is for images that leave SMs idle anyway.
// Slot NT is the thread that does not exist (zeros, read beyond the tile).
template <int A, int MODE>
__device__ __forceinline__ void zb_step(f32x2 (&xE)[ZB_ROWS], f32x2 (&xO)[ZB_ROWS],
                                        const f32x2 (&bE)[ZB_ROWS], const f32x2 (&bO)[ZB_ROWS],
                                        unsigned char* sm, int NS, int t, int tu, int td, int tl, int tr,
                                        f32x2 cw, f32x2 c1, f32x2 cb) {
  // MODE 0: first step, x = cb b; 1: x = cw S + c1 x + cb b; 2: x = cw S + c1 x + b.
  // Edges of one colour: [top, bottom] pairs, then [left, right] columns of ZB_ROWS / 2 values
  const int colour = NS * 32;
  float le[ZB_ROWS / 2], ri[ZB_ROWS / 2];
  f32x2 up = 0, dn = 0;
  if constexpr (MODE != 0) {
    const unsigned char* o = sm + (1 - A) * colour;
    const f32x2* rows = reinterpret_cast<const f32x2*>(o);
    const float2* cols = reinterpret_cast<const float2*>(o + (size_t)NS * 16);
    up = rows[NS + tu];                      // bottom row of the block above
    dn = rows[td];                           // top row of the block below
    const float2 l = cols[NS + tl], r = cols[tr];
    le[0] = l.x; le[1] = l.y;
    ri[0] = r.x; ri[1] = r.y;
  }
  float eL[ZB_ROWS / 2], eR[ZB_ROWS / 2];
#pragma unroll
  for (int i = 0; i < ZB_ROWS; ++i) {
    const int iu = i > 0 ? i - 1 : 0, id = i < ZB_ROWS - 1 ? i + 1 : i;
    if ((i + A) % 2 == 0) {
      const f32x2 bb = MODE == 2 ? bE[i] : mul2(bE[i], cb);
      if constexpr (MODE == 0) {
        xE[i] = bb;
      } else {
        const float o0 = lo2(xO[i]), o1 = hi2(xO[i]);
        const f32x2 s = add2(add2(i > 0 ? xE[iu] : up, i < ZB_ROWS - 1 ? xE[id] : dn), pk2(le[i / 2] + o0, o0 + o1));
        xE[i] = fma2(s, cw, fma2(xE[i], c1, bb));
      }
      eL[i / 2] = lo2(xE[i]);
    } else {
      const f32x2 bb = MODE == 2 ? bO[i] : mul2(bO[i], cb);
      if constexpr (MODE == 0) {
        xO[i] = bb;
      } else {
        const float e0 = lo2(xE[i]), e1 = hi2(xE[i]);
        const f32x2 s = add2(add2(i > 0 ? xO[iu] : up, i < ZB_ROWS - 1 ? xO[id] : dn), pk2(e0 + e1, e1 + ri[i / 2]));
        xO[i] = fma2(s, cw, fma2(xO[i], c1, bb));
      }
      eR[i / 2] = hi2(xO[i]);
    }
  }
  unsigned char* w = sm + A * colour;
  f32x2* rows = reinterpret_cast<f32x2*>(w);
  float2* cols = reinterpret_cast<float2*>(w + (size_t)NS * 16);
  rows[t] = A == 0 ? xE[0] : xO[0];
  rows[NS + t] = A == 0 ? xO[ZB_ROWS - 1] : xE[ZB_ROWS - 1];
  cols[t] = make_float2(eL[0], eL[1]);
  cols[NS + t] = make_float2(eR[0], eR[1]);
  __syncthreads();
}

// Predicated load of the KC classes [k0, k0 + KC) of a quad (or of a dense pixel): zeros where
// `ok` is false (the address is then not read).
template <int KC>
__device__ __forceinline__ void ldk_if(float (&v)[KC], const float* p, bool ok) {
  if constexpr (KC == 4) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.s32 p, %5, 0;\n mov.f32 %0, 0f00000000;\n"
        " mov.f32 %1, 0f00000000;\n mov.f32 %2, 0f00000000;\n mov.f32 %3, 0f00000000;\n"
        " @p ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];\n}\n"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
        : "l"(p), "r"((int)ok));
  } else if constexpr (KC == 2) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.s32 p, %3, 0;\n mov.f32 %0, 0f00000000;\n"
        " mov.f32 %1, 0f00000000;\n @p ld.global.nc.v2.f32 {%0, %1}, [%2];\n}\n"
        : "=f"(v[0]), "=f"(v[1])
        : "l"(p), "r"((int)ok));
  } else {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.s32 p, %2, 0;\n mov.f32 %0, 0f00000000;\n"
        " @p ld.global.nc.f32 %0, [%1];\n}\n"
        : "=f"(v[0])
        : "l"(p), "r"((int)ok));
  }
}

// DENSE: 0 tile partials, 1 dense rhs whose KC classes are one aligned vector, 2 value by value.
template <int KC, int DENSE>
__global__ void __launch_bounds__(ZB_THREADS) k_zblock(const ZlArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int2 rowof[ZB_MAXSIDE], colof[ZB_MAXSIDE];  // offsets of the covers (or of the pixel)
  const int t = threadIdx.x, NT = blockDim.x, NS = NT + 1;
  const int ngc = (a.K + KC - 1) / KC;           // class groups
  const int g = blockIdx.x % ngc, tile = blockIdx.x / ngc;
  const int ty = tile / a.p.nx, tx = tile - ty * a.p.nx;
  const int y0 = (int)(((long long)ty * a.H) / a.p.ny), y1 = (int)(((long long)(ty + 1) * a.H) / a.p.ny);
  const int x0 = (int)(((long long)tx * a.W) / a.p.nx), x1 = (int)(((long long)(tx + 1) * a.W) / a.p.nx);
  const int NBX = a.p.nbx, NBY = a.p.nby, TW = 4 * NBX, TH = NBY * ZB_ROWS;
  const int k0 = g * KC;
  // the tile's rhs, KC classes a pixel, goes into [class][row][column] planes (padded by one
  // quad so that the planes start on different banks); the offsets of its rows and columns are
  // set up before the wait for the previous kernel
  float* st = reinterpret_cast<float*>(smem_raw);
  const int plane = TW * TH + 4;
  for (int r = t; r < TH; r += NT) {
    const int gy = wrap_idx(y0 - ZL_HALO + r, a.H);
    rowof[r] = DENSE == 0 ? __ldg(reinterpret_cast<const int2*>(a.offY) + gy) : make_int2(gy * a.W, -1);
  }
  for (int c = t; c < TW; c += NT) {
    const int gx = wrap_idx(x0 - ZL_HALO + c, a.W);
    int2 o = make_int2(gx, -1);
    if constexpr (DENSE == 0) {
      const int2 cx = __ldg(reinterpret_cast<const int2*>(a.covX) + gx);
      const int pl = a.EHmax * a.EWmax, q = k0 >> 2;
      o.x = ((cx.x >> 16) * a.ng + q) * pl + (cx.x & 0xffff);
      if (cx.y >= 0) o.y = ((cx.y >> 16) * a.ng + q) * pl + (cx.y & 0xffff);
    }
    colof[c] = o;
  }
  const uint32_t mgw = (uint32_t)((0x100000000ULL + (unsigned)TW - 1) / (unsigned)TW);
  __syncthreads();
  pdl_wait();  // the rhs comes from the previous kernel
  // a thread's block holds 16 values, and so does its share of the loads: all in flight at once
  constexpr int U = 4 * ZB_ROWS / KC;
  for (int p0 = t; p0 < TW * TH; p0 += U * NT) {
    float v[U][KC], h[U][KC], u[U][KC], w[U][KC];
#pragma unroll
    for (int e = 0; e < U; ++e) {
      const int p = p0 + e * NT;
      const bool in = p < TW * TH;
      const int r = in ? (int)__umulhi((uint32_t)p, mgw) : 0;
      const int2 ro = rowof[r], co = colof[in ? p - r * TW : 0];
      if constexpr (DENSE == 0) {
        const float* P = a.P + (k0 & 3);
        const bool hx = co.y >= 0 && in, hy = ro.y >= 0 && in;
        ldk_if<KC>(v[e], P + 4 * (long long)(ro.x + co.x), in);
        ldk_if<KC>(h[e], P + 4 * (long long)(ro.x + co.y), hx);
        ldk_if<KC>(u[e], P + 4 * (long long)(ro.y + co.x), hy);
        ldk_if<KC>(w[e], P + 4 * (long long)(ro.y + co.y), hy && hx);
      } else {
        const float* s = a.src + (size_t)(ro.x + co.x) * a.K + k0;
        if constexpr (DENSE == 1) {
          ldk_if<KC>(v[e], s, in);
        } else {
#pragma unroll
          for (int j = 0; j < KC; ++j) {
            float one[1];
            ldk_if<1>(one, s + j, in && k0 + j < a.K);
            v[e][j] = one[0];
          }
        }
      }
    }
#pragma unroll
    for (int e = 0; e < U; ++e) {
      const int p = p0 + e * NT;
      if (p < TW * TH) {
#pragma unroll
        for (int j = 0; j < KC; ++j)
          st[j * plane + p] = (DENSE == 0 ? ((v[e][j] + h[e][j]) + u[e][j]) + w[e][j] : v[e][j]) * a.q.bs;
      }
    }
  }
  pdl_trigger();
  const int blk = t / KC, kc = t - blk * KC;
  const int by = blk / NBX, bx = blk - by * NBX;
  const bool in = by < NBY;
  const int rowt = KC * NBX;
  const int tu = in && by > 0 ? t - rowt : NT, td = in && by < NBY - 1 ? t + rowt : NT;
  const int tl = in && bx > 0 ? t - KC : NT, tr = in && bx < NBX - 1 ? t + KC : NT;
  __syncthreads();
  f32x2 xE[ZB_ROWS], xO[ZB_ROWS], bE[ZB_ROWS], bO[ZB_ROWS];
  const float* sb = st + kc * plane + (in ? by : 0) * ZB_ROWS * TW + 4 * bx;
#pragma unroll
  for (int i = 0; i < ZB_ROWS; ++i) {
    const float4 v = *reinterpret_cast<const float4*>(sb + i * TW);
    bE[i] = pk2(v.x, v.z);
    bO[i] = pk2(v.y, v.w);
    xE[i] = xO[i] = 0;
  }
  __syncthreads();                               // the planes become the edge slots
  if (t < 8) reinterpret_cast<f32x2*>(smem_raw)[t * NS + NT] = 0;  // the missing neighbour's edges
  zb_step<0, 0>(xE, xO, bE, bO, smem_raw, NS, t, tu, td, tl, tr, 0, 0, pk2(a.q.b0));
  static_assert(ZL_EARLY == 2 && (ZL_STEPS - 1 - ZL_EARLY) % 2 == 0, "step schedule");
  zb_step<1, 1>(xE, xO, bE, bO, smem_raw, NS, t, tu, td, tl, tr, pk2(a.q.cw[0]), pk2(a.q.c1[0]), pk2(a.q.cb[0]));
  zb_step<0, 1>(xE, xO, bE, bO, smem_raw, NS, t, tu, td, tl, tr, pk2(a.q.cw[1]), pk2(a.q.c1[1]), pk2(a.q.cb[1]));
  const f32x2 cw = pk2(a.q.cw[ZL_EARLY]), c1 = pk2(a.q.c1[ZL_EARLY]);
#pragma unroll 1
  for (int s = 0; s < (ZL_STEPS - 1 - ZL_EARLY) / 2; ++s) {
    zb_step<1, 2>(xE, xO, bE, bO, smem_raw, NS, t, tu, td, tl, tr, cw, c1, 0);
    zb_step<0, 2>(xE, xO, bE, bO, smem_raw, NS, t, tu, td, tl, tr, cw, c1, 0);
  }
  if (!in || k0 + kc >= a.K) return;
  const int yb = y0 - ZL_HALO + ZB_ROWS * by, xb = x0 - ZL_HALO + 4 * bx;
  float* zp = a.z + ((long long)yb * a.W + xb) * a.K + k0 + kc;
#pragma unroll
  for (int i = 0; i < ZB_ROWS; ++i) {
    if (yb + i >= y0 && yb + i < y1) {
      const float o[4] = {lo2(xE[i]), lo2(xO[i]), hi2(xE[i]), hi2(xO[i])};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (xb + j >= x0 && xb + j < x1) zp[((long long)i * a.W + j) * a.K] = o[j];
    }
  }
}

template <int KC, int DENSE>
static cudaError_t zb_launch(const ZlArgs& a, cudaStream_t st) {
  static SmemGrants grant;
  const size_t smem = zb_smem(a.p);
  const cudaError_t e = grant_smem(k_zblock<KC, DENSE>, smem, grant);
  if (e != cudaSuccess) return e;
  // small CTAs share SMs with the sweep before and after them: its carve-out (two sizes measured; 100 x 90, K = 4:
  // 17.8 -> 12.0 us per iteration; 145 x 145, K = 16, whose 512 threads take an SM each and use
  // the L1: 20.3 us without, 21.3 with)
  return launch_pdl_carve(a.p.threads <= 256, k_zblock<KC, DENSE>, dim3(a.p.nx * a.p.ny * ((a.K + KC - 1) / KC)), dim3(a.p.threads), smem, st, a);
}
template <int KC>
static cudaError_t zb_launch_src(const ZlArgs& a, cudaStream_t st) {
  if (!a.src) return zb_launch<KC, 0>(a, st);
  if (a.K % KC == 0 && reinterpret_cast<uintptr_t>(a.src) % (4 * KC) == 0) return zb_launch<KC, 1>(a, st);
  return zb_launch<KC, 2>(a, st);
}

template <int MODE, bool VEC>
static cudaError_t zs_launch(const ZlArgs& a, cudaStream_t st) {
  static SmemGrants grant;
  constexpr size_t smem = zs_smem<MODE>();
  const cudaError_t e = grant_smem(k_zstream<MODE, VEC>, smem, grant);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_zstream<MODE, VEC>, dim3(a.p.nx * a.p.ny * a.ng), dim3(128), smem, st, a);
}

cudaError_t launch_zlocal(const ZlArgs& a0, cudaStream_t st) {
  ZlArgs a = a0;
  a.ng = (a.K + 3) / 4;
  if (a.p.kc == 1) return zb_launch_src<1>(a, st);
  if (a.p.kc == 2) return zb_launch_src<2>(a, st);
  if (a.p.kc == 4) return zb_launch_src<4>(a, st);
  const bool vec = a.K % 4 == 0 && (reinterpret_cast<uintptr_t>(a.z) & 15) == 0;
  const bool svec = a.K % 4 == 0 && (reinterpret_cast<uintptr_t>(a.src) & 15) == 0;
  if (!a.src) return vec ? zs_launch<0, true>(a, st) : zs_launch<0, false>(a, st);
  if (svec) return vec ? zs_launch<1, true>(a, st) : zs_launch<1, false>(a, st);
  return vec ? zs_launch<2, true>(a, st) : zs_launch<2, false>(a, st);
}

}  // namespace sgs
