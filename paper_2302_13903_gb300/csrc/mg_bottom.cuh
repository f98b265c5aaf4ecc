// mg_bottom.cuh -- one V(1,1) cycle on the levels of at most 16^3 cells of a
// batched grid, by one CTA in shared memory (device code of mg_batch.cu).
//
// The cycle is a chain of some 25 passes over at most 4096 cells, so its time
// is the latency of a pass.  Sizes and the kind of rule are known at compile
// time; a level's two colours are apart, so that an item (W cells of one colour
// of a row, W = 4 on the 16^3 and 8^3 levels) reads whole 16-byte words without
// bank conflicts (planes of 16^3 and 8^3 are padded); the levels of 4^3 and
// below are one warp's, which meets no block barrier.  Against block-strided
// loops over single cells with run-time sizes and an FP64 set-up by one thread,
// 12-20 launches of which are in a solve (GB300, ms): 256 grids of 16^3 1.38 ->
// 0.99, one of 128^3 1.30 -> 1.13, 512 of 16-128 23.8 -> 22.8.
//
// What a cell computes does not depend on the CTA's size, so every caller gets
// the same bits.
#pragma once

#include <cuda_runtime.h>

#include "mg_device.cuh"
#include "mg_internal.h"

namespace mg {
namespace bottom {

constexpr int kTopN = 16;  // cells a side of the largest level

// The top level in global memory (natural order), rule and coefficients:
// u <- cu u + cs sum_nb + cf f, 1 / h^2 for defects (of the top level: level by
// level down, cf grows and ih2 falls by exactly 4).
struct Args {
  float* u;
  const float* f;
  bool zero;  // u starts at 0
  float sgn;  // ghost across a wall: sgn times the cell (fixed -1, zero gradient 1)
  float cu, cs, cf, ih2;
};

// One colour of a level with N cells a side: cell m of row (j, k) at j R + k S + m.
template <int N>
struct Lev {
  static constexpr int W = N >= 8 ? 4 : N / 2;  // cells of a colour per item
  static constexpr int H = N / 2 / W;           // items per row
  static constexpr int R = N / 2;               // floats between rows
  static constexpr int S = N == 16 ? 144 : N == 8 ? 48 : N * N / 2;  // between planes
  static constexpr int SIZE = N * S;
  static constexpr int ITEMS = N * N * H;
};
// uR, uB, fR, fB of the levels, largest first.
template <int N>
struct Offset {
  static constexpr int v = Offset<2 * N>::v + 4 * Lev<2 * N>::SIZE;
};
template <>
struct Offset<kTopN> {
  static constexpr int v = 0;
};
constexpr size_t kBytes = sizeof(float) * (Offset<1>::v + 4);

struct Block {
  static __device__ __forceinline__ int id() { return threadIdx.x; }
  static __device__ __forceinline__ int size() { return blockDim.x; }
  static __device__ __forceinline__ void sync() { __syncthreads(); }
};
struct Warp {
  static __device__ __forceinline__ int id() { return threadIdx.x; }  // warp 0
  static __device__ __forceinline__ int size() { return 32; }
  static __device__ __forceinline__ void sync() { __syncwarp(); }
};

template <int W>
__device__ __forceinline__ void load(float (&v)[W], const float* p) {
  if constexpr (W == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
  } else {
#pragma unroll
    for (int m = 0; m < W; ++m) v[m] = p[m];
  }
}
template <int W>
__device__ __forceinline__ void store(float* p, const float (&v)[W]) {
  if constexpr (W == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int m = 0; m < W; ++m) p[m] = v[m];
  }
}

// Item t of a level: cells [h W, (h + 1) W) of a colour of row (j, k).  The four
// rows of a coarse row, and their H items, are neighbouring lanes.
template <int N>
struct Item {
  int h, j, k;
  bool e;  // red is the odd cell of each pair
  int o;   // offset of the item's cells in a colour
  __device__ __forceinline__ explicit Item(int t) {
    constexpr int H = Lev<N>::H;
    h = t & (H - 1);
    t /= H;
    j = 2 * ((t >> 2) & (N / 2 - 1)) + (t & 1);
    k = 2 * ((t >> 2) / (N / 2)) + ((t >> 1) & 1);
    e = (j ^ k) & 1;
    o = j * Lev<N>::R + k * Lev<N>::S + h * Lev<N>::W;
  }
};

// The rows y-, y+, z-, z+ of an item: offset of their cells, or for a wall of
// the item's own with the ghost's sign.
template <int N, bool PER>
struct Rows {
  int o[4];
  bool wall[4];
  __device__ __forceinline__ explicit Rows(const Item<N>& it) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bool hi = q & 1;
      const int x = q < 2 ? it.j : it.k, d = q < 2 ? Lev<N>::R : Lev<N>::S;
      const bool end = x == (hi ? N - 1 : 0);
      wall[q] = !PER && end;
      const int to = end ? (PER ? (hi ? 1 - N : N - 1) : 0) : (hi ? 1 : -1);
      o[q] = it.o + to * d;
    }
  }
};

// The cell of a colour next to the item's along x, on the high or low side
// (`own`: the item's cell at that end, whose ghost stands in at a wall).
template <int N, bool PER>
__device__ __forceinline__ float beyond(const float* c, const Item<N>& it, bool up, float own,
                                        float sgn) {
  constexpr int W = Lev<N>::W, H = Lev<N>::H;
  const bool end = it.h == (up ? H - 1 : 0);
  if (!PER && end) return sgn * own;
  return c[it.o + (up ? (end ? W - N / 2 : W) : (end ? N / 2 - 1 : -1))];
}

// One colour of SMOOTH (own) from the other (oth).
template <int N, bool PER, typename G>
__device__ __forceinline__ void sweep(float* own, const float* oth, const float* f, bool red,
                                      float sgn, float cu, float cs, float cf) {
  constexpr int W = Lev<N>::W;
  for (int t = G::id(); t < Lev<N>::ITEMS; t += G::size()) {
    const Item<N> it(t);
    const Rows<N, PER> rw(it);
    float a[W], n[W], g[W], s[W];
    load<W>(a, own + it.o);
    load<W>(n, oth + it.o);
    load<W>(g, f + it.o);
    const bool up = red == it.e;  // the cell outside the pair is on the high side
    const float x = beyond<N, PER>(oth, it, up, up ? a[W - 1] : a[0], sgn);
#pragma unroll
    for (int m = 0; m < W; ++m)
      s[m] = n[m] + (up ? (m + 1 < W ? n[m + 1 < W ? m + 1 : 0] : x) : (m > 0 ? n[m > 0 ? m - 1 : 0] : x));
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float v[W];
      load<W>(v, (PER || !rw.wall[q] ? oth : own) + rw.o[q]);
      const float w = PER || !rw.wall[q] ? 1.f : sgn;
#pragma unroll
      for (int m = 0; m < W; ++m) s[m] = fmaf(w, v[m], s[m]);
    }
#pragma unroll
    for (int m = 0; m < W; ++m) a[m] = fmaf(cs, s[m], fmaf(cu, a[m], cf * g[m]));
    store<W>(own + it.o, a);
  }
  G::sync();
}

// SMOOTH (red first); `first`: u starts at 0.
template <int N, bool PER, typename G>
__device__ __forceinline__ void smooth(float* sm, bool first, const Args& a, float cf) {
  constexpr int W = Lev<N>::W, Z = Lev<N>::SIZE;
  float *uR = sm + Offset<N>::v, *uB = uR + Z, *fR = uB + Z, *fB = fR + Z;
  if (first) {
    for (int t = G::id(); t < Lev<N>::ITEMS; t += G::size()) {
      const Item<N> it(t);
      float g[W], z[W];
      load<W>(g, fR + it.o);
#pragma unroll
      for (int m = 0; m < W; ++m) {
        g[m] = cf * g[m];
        z[m] = 0.f;
      }
      store<W>(uR + it.o, g);
      store<W>(uB + it.o, z);
    }
    G::sync();
  } else {
    sweep<N, PER, G>(uR, uB, fR, true, a.sgn, a.cu, a.cs, cf);
  }
  sweep<N, PER, G>(uB, uR, fB, false, a.sgn, a.cu, a.cs, cf);
}

// Cell I of coarse row (J, K) of a level's colours c (red) and c + SIZE.
template <int N>
__device__ __forceinline__ int at(int I, int J, int K) {
  if constexpr (N == 1) return 0;
  else return ((I ^ J ^ K) & 1 ? Lev<N>::SIZE : 0) + J * Lev<N>::R + K * Lev<N>::S + (I >> 1);
}

// f of the next level: the mean defect of the eight children.  An item sums
// its W pairs, four lanes the rows of a coarse row.
template <int N, bool PER, typename G>
__device__ __forceinline__ void restrict_defect(float* sm, const Args& a, float ih2) {
  constexpr int W = Lev<N>::W, H = Lev<N>::H, Z = Lev<N>::SIZE, NC = N / 2;
  const float *uR = sm + Offset<N>::v, *uB = uR + Z, *fR = uB + Z, *fB = fR + Z;
  float* fc = sm + Offset<NC>::v + (NC > 1 ? 2 * Lev<NC>::SIZE : 1);
  for (int t = G::id(); t < Lev<N>::ITEMS; t += G::size()) {
    const Item<N> it(t);
    const Rows<N, PER> rw(it);
    float r[W], b[W], g[W], h[W], d[W];
    load<W>(r, uR + it.o);
    load<W>(b, uB + it.o);
    load<W>(g, fR + it.o);
    load<W>(h, fB + it.o);
    // the cells left and right of each pair: left the colour of its odd cell,
    // right the colour of its even cell
    const float xl = beyond<N, PER>(it.e ? uR : uB, it, false, it.e ? b[0] : r[0], a.sgn);
    const float xr = beyond<N, PER>(it.e ? uB : uR, it, true, it.e ? r[W - 1] : b[W - 1], a.sgn);
#pragma unroll
    for (int m = 0; m < W; ++m) {
      const float l = m > 0 ? (it.e ? r[m > 0 ? m - 1 : 0] : b[m > 0 ? m - 1 : 0]) : xl;
      const float u = m + 1 < W ? (it.e ? b[m + 1 < W ? m + 1 : 0] : r[m + 1 < W ? m + 1 : 0]) : xr;
      d[m] = fmaf(-5.f, r[m] + b[m], l + u);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float v[W], w[W];
      load<W>(v, uR + rw.o[q]);
      load<W>(w, uB + rw.o[q]);
      const float sg = PER || !rw.wall[q] ? 1.f : a.sgn;
#pragma unroll
      for (int m = 0; m < W; ++m) d[m] = fmaf(sg, v[m] + w[m], d[m]);
    }
    // the lanes of a coarse row; ITEMS and every group size are multiples of 4 H
    const unsigned mask = ((1u << (4 * H)) - 1) << (threadIdx.x & 31 & ~(4 * H - 1));
#pragma unroll
    for (int m = 0; m < W; ++m) {
      d[m] = fmaf(-ih2, d[m], g[m] + h[m]);
      d[m] += __shfl_xor_sync(mask, d[m], H);
      d[m] += __shfl_xor_sync(mask, d[m], 2 * H);
    }
    if (!((it.j | it.k) & 1)) {
#pragma unroll
      for (int m = 0; m < W; ++m)
        fc[at<NC>(it.h * W + m, it.j >> 1, it.k >> 1)] = 0.125f * d[m];
    }
  }
  G::sync();
}

// u += trilinear(u of the next level).
template <int N, bool PER, typename G>
__device__ __forceinline__ void prolong_add(float* sm, const Args& a) {
  constexpr int W = Lev<N>::W, Z = Lev<N>::SIZE, NC = N / 2;
  float *uR = sm + Offset<N>::v, *uB = uR + Z;
  const float* c = sm + Offset<NC>::v;
  for (int t = G::id(); t < Lev<N>::ITEMS; t += G::size()) {
    const Item<N> it(t);
    // coarse index x + d, wrapped, or the edge cell with the ghost's sign
    auto near = [&](int x, int d, float& s) {
      const int y = x + d;
      s = 1.f;
      if (y >= 0 && y < NC) return y;
      if (PER) return y & (NC - 1);
      s = a.sgn;
      return x;
    };
    float sy, sz, sl, sr;
    const int J = it.j >> 1, K = it.k >> 1, I0 = it.h * W;
    const int J2 = near(J, it.j & 1 ? 1 : -1, sy), K2 = near(K, it.k & 1 ? 1 : -1, sz);
    const int Il = near(I0, -1, sl), Ir = near(I0 + W - 1, 1, sr);
    float v[W + 2];  // the coarse rows' mean at I0 - 1 .. I0 + W, times 16
#pragma unroll
    for (int m = 0; m < W + 2; ++m) {
      const int I = m == 0 ? Il : m == W + 1 ? Ir : I0 + m - 1;
      float x = 9.f * c[at<NC>(I, J, K)];
      x = fmaf(3.f * sy, c[at<NC>(I, J2, K)], x);
      x = fmaf(3.f * sz, c[at<NC>(I, J, K2)], x);
      v[m] = fmaf(sy * sz, c[at<NC>(I, J2, K2)], x);
    }
    v[0] *= sl;
    v[W + 1] *= sr;
    float r[W], b[W];
    load<W>(r, uR + it.o);
    load<W>(b, uB + it.o);
#pragma unroll
    for (int m = 0; m < W; ++m) {
      const float lo = fmaf(3.f, v[m + 1], v[m]), hi = fmaf(3.f, v[m + 1], v[m + 2]);
      r[m] = fmaf(0.015625f, it.e ? hi : lo, r[m]);
      b[m] = fmaf(0.015625f, it.e ? lo : hi, b[m]);
    }
    store<W>(uR + it.o, r);
    store<W>(uB + it.o, b);
  }
  G::sync();
}

// The cycle on the level of N cells a side and those below.
template <int N, bool PER, typename G>
__device__ void levels(float* sm, bool first, const Args& a, float cf, float ih2) {
  if constexpr (N == 1) {  // one cell, exactly: (2 sgn - 2) 3 u = h^2 f, or 0 where singular
    if (G::id() == 0) {
      float* u = sm + Offset<1>::v;
      u[0] = !PER && a.sgn < 0.f ? u[1] * (-1.f / (12.f * ih2)) : 0.f;
    }
    G::sync();
  } else {
    smooth<N, PER, G>(sm, first, a, cf);
    restrict_defect<N, PER, G>(sm, a, ih2);
    if constexpr (N == 8) {  // the levels of 4^3 and below: one warp
      if (threadIdx.x < 32) levels<4, PER, Warp>(sm, true, a, 4.f * cf, 0.25f * ih2);
      __syncthreads();
    } else {
      levels<N / 2, PER, G>(sm, true, a, 4.f * cf, 0.25f * ih2);
    }
    prolong_add<N, PER, G>(sm, a);
    smooth<N, PER, G>(sm, false, a, cf);
  }
}

// f (and u) of the top level into its colours, the cycle, u back.
template <int N, bool PER>
__device__ void run(float* sm, const Args& a) {
  constexpr int W = Lev<N>::W, Z = Lev<N>::SIZE;
  float *uR = sm + Offset<N>::v, *uB = uR + Z, *fR = uB + Z, *fB = fR + Z;
  auto split = [&](const float* p, const Item<N>& it, float* red, float* blk) {
    float lo[W], hi[W], r[W], b[W];
    p += ((size_t)it.k * N + it.j) * N + 2 * W * it.h;
    load<W>(lo, p);
    load<W>(hi, p + W);
#pragma unroll
    for (int m = 0; m < W; ++m) {
      const float x = 2 * m < W ? lo[2 * m < W ? 2 * m : 0] : hi[2 * m < W ? 0 : 2 * m - W];
      const float y = 2 * m + 1 < W ? lo[2 * m + 1 < W ? 2 * m + 1 : 0]
                                    : hi[2 * m + 1 < W ? 0 : 2 * m + 1 - W];
      r[m] = it.e ? y : x;
      b[m] = it.e ? x : y;
    }
    store<W>(red + it.o, r);
    store<W>(blk + it.o, b);
  };
  for (int t = threadIdx.x; t < Lev<N>::ITEMS; t += blockDim.x) {
    const Item<N> it(t);
    split(a.f, it, fR, fB);
    if (!a.zero) split(a.u, it, uR, uB);
  }
  __syncthreads();
  levels<N, PER, Block>(sm, a.zero, a, a.cf, a.ih2);
  for (int t = threadIdx.x; t < Lev<N>::ITEMS; t += blockDim.x) {
    const Item<N> it(t);
    float r[W], b[W], v[2 * W];
    load<W>(r, uR + it.o);
    load<W>(b, uB + it.o);
#pragma unroll
    for (int m = 0; m < W; ++m) {
      v[2 * m] = it.e ? b[m] : r[m];
      v[2 * m + 1] = it.e ? r[m] : b[m];
    }
    float* p = a.u + ((size_t)it.k * N + it.j) * N + 2 * W * it.h;
    float lo[W], hi[W];
#pragma unroll
    for (int m = 0; m < W; ++m) {
      lo[m] = v[m];
      hi[m] = v[W + m];
    }
    store<W>(p, lo);
    store<W>(p + W, hi);
  }
}

// The cycle from a top level of n = 2, 4, 8 or 16 cells a side; the CTA has at
// least 32 threads, a multiple of 8.
__device__ __forceinline__ void vcycle(int n, bool per, float* sm, const Args& a) {
  switch (n) {
    case 16: per ? run<16, true>(sm, a) : run<16, false>(sm, a); break;
    case 8: per ? run<8, true>(sm, a) : run<8, false>(sm, a); break;
    case 4: per ? run<4, true>(sm, a) : run<4, false>(sm, a); break;
    default: per ? run<2, true>(sm, a) : run<2, false>(sm, a); break;
  }
}

}  // namespace bottom
}  // namespace mg
