// mg_fx64.cu -- the finest level of the FP64 path in exact 64-bit fixed point.
//
// An SM issues two FP64 operations per clock, so a V(1,1) cycle's 25-30 FP64
// operations per cell take several times as long as its bytes.  Here phi and
// h^2 f of the finest level are 64-bit integers scaled by 2^S with |phi| <
// 2^55: a quantum of at most 2^-54 max|phi|, against the 2^-53 of a double.
// With U and F those integers,
//   R = (sum of the six neighbours of U) - 6 U - F       (exactly)
//   SMOOTH: U += round(R omega / 6)                      (Eqs. rbsor1-rbsor2)
//   defect: f - L u = -R / (h^2 2^S)                     (Eq. defect)
// so neighbour sums and defects carry no rounding at all, and one update rounds
// once.  omega / 6 is a 64-bit fraction.  A face's value b enters the ghost 2 b - u as a
// constant and is folded into F (F - round(2 b 2^S)) when F is formed, so the
// sweeps run the homogeneous rule.
//
// Two z-marching kernels, like the FP32 legs: down = one SMOOTH and the
// restricted defect, up = the prolonged correction and one SMOOTH.  A CTA
// owns 64 x 16 columns; a thread has a pair of cells along x, one of each
// colour in every plane, so each half-step updates one cell per thread.  What
// it reads of its neighbours is the other colour of the same plane: its own
// pair's cell (a register), and through shared memory the next pair's along x
// and the rows above and below; the planes above and below are its own
// registers.  Half-step s of plane p runs one step after half-step s of plane
// p - 1 and reads only what the step before wrote: one barrier per plane.
// Planes arrive by 16-byte cp.async into a ring that each thread fills and
// reads back itself.  A CTA recomputes its halo (3 cells on the down leg, 2 on
// the up leg), so CTAs never wait on one another.
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>

#include "mg_convert.cuh"
#include "mg_device.cuh"
#include "mg_internal.h"

namespace mg {
namespace {

constexpr int TX = 64, TY = 16;
constexpr int kRing = 4;  // planes of the cp.async ring

// omega / 6 = (hi + lo / 2^32) / 2^32.
struct Weight {
  int hi, lo;
};

struct Fx64Args {
  const long long* u_in;
  long long* u_out;
  const long long* F;
  Grid g;
  int fk;        // kinds of the faces (homogeneous), 2 bits each
  int cz;        // planes per CTA (even)
  Weight w;
  double* norm;  // per-CTA sum of R^2: red cells of u_in (down), black cells of u_out (up)
  double* fc;           // down: coarse right-hand side, -sum of R / 8
  long long* psum;      // down: per-CTA exact sum of u_in, (hi, lo) pairs
  const long long* ec;  // up: coarse correction on the integer grid
  int* flag;            // |U| passed 2^59
};

// round(R w), halves up, for w = (hi + lo / 2^32) / 2^32 < 1/3 and |R| < 2^63:
// the product's part below 2^-32 of lo's weight (2^-32 of a quantum) is left
// out; the middle terms stay below 2^63 together.
__device__ __forceinline__ long long weigh(long long R, Weight w) {
  const long long mid = (long long)((unsigned long long)(unsigned)R * (unsigned)w.hi + 0x80000000ull) +
                        (long long)(int)(R >> 32) * w.lo;
  return (long long)(int)(R >> 32) * w.hi + (mid >> 32);
}

__device__ __forceinline__ void cp16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// The window of a CTA: its tile and a halo of HX cells and HY rows.
template <int HX, int HY>
struct Win {
  static constexpr int PW = (TX + 2 * HX) / 2;  // pairs per row
  static constexpr int RH = TY + 2 * HY;
  static constexpr int NT = PW * RH;
  static constexpr int PAD = PW + 1;  // so that every neighbour index is in range
  static constexpr int PLANE = NT + 2 * PAD;
};
using Down = Win<4, 3>;
using Up = Win<2, 2>;

struct Ring {
  template <int NT>
  struct Of {
    longlong2 u[kRing][NT];
    longlong2 f[kRing][NT];
  };
};

// What a thread knows about its pair of columns.  Column P is the one that is
// red in even planes, column Q the one that is red in odd planes.
struct Pair {
  int i0, j;       // cells (i0, j) and (i0 + 1, j), wrapped into the level
  bool valid;      // inside the level
  bool tile;       // written by this CTA
  bool swap;       // P is cell i0 + 1
  int xo;          // pair offset of P's neighbour outside the pair (Q's is -xo)
  // walls (never with periodic axes): sign of the ghost, 0 where there is none
  int wxp, wxq, wyl, wyh;
};

__device__ __forceinline__ int wall_sign(int fk, int q) {
  const int kind = (fk >> (2 * q)) & 3;
  return kind == BC_PERIODIC ? 0 : kind == BC_ZEROGRAD ? 1 : -1;
}

template <typename W, int HX, int HY>
__device__ __forceinline__ Pair make_pair_of(const Fx64Args& a, int t) {
  Pair p;
  const int pm = t % W::PW, pr = t / W::PW;
  int i = (int)blockIdx.x * TX + 2 * pm - HX, j = (int)blockIdx.y * TY + pr - HY;
  p.tile = pm >= HX / 2 && pm < HX / 2 + TX / 2 && pr >= HY && pr < HY + TY;
  const bool px = (a.fk & 3) == BC_PERIODIC, py = ((a.fk >> 4) & 3) == BC_PERIODIC;
  p.valid = (px || (i >= 0 && i < a.g.nx)) && (py || (j >= 0 && j < a.g.ny));
  p.swap = j & 1;
  p.xo = p.swap ? 1 : -1;
  const int xl = i == 0 ? wall_sign(a.fk, 0) : 0, xh = i + 2 == a.g.nx ? wall_sign(a.fk, 1) : 0;
  p.wxp = p.swap ? xh : xl;
  p.wxq = p.swap ? xl : xh;
  p.wyl = j == 0 ? wall_sign(a.fk, 2) : 0;
  p.wyh = j == a.g.ny - 1 ? wall_sign(a.fk, 3) : 0;
  // a level may be narrower than the window's reach: wrap by remainder
  i = (i + 2 * a.g.nx) % a.g.nx;
  j = (j + 2 * a.g.ny) % a.g.ny;
  p.i0 = i;
  p.j = j;
  if (!p.valid) p.i0 = p.j = 0;
  return p;
}

__device__ __forceinline__ long long signed_by(int s, long long v) { return s < 0 ? -v : v; }

// Sum of the six neighbours of a cell holding `self` whose colour's other
// values of the plane are in `o` (at this thread's index); `mate` is the
// pair's other cell, xo the offset of the neighbour outside the pair.
template <bool WALLS, int PW>
__device__ __forceinline__ long long sum6(const long long* o, long long self, long long mate, int xo,
                                          int wx, const Pair& p, long long zl, long long zh, int wzl,
                                          int wzh) {
  long long x = o[xo], yl = o[-PW], yh = o[PW];
  if (WALLS) {
    if (wx) x = signed_by(wx, self);
    if (p.wyl) yl = signed_by(p.wyl, self);
    if (p.wyh) yh = signed_by(p.wyh, self);
    if (wzl) zl = signed_by(wzl, self);
    if (wzh) zh = signed_by(wzh, self);
  }
  return ((mate + x) + (yl + yh)) + (zl + zh);
}

__device__ __forceinline__ bool too_large(long long v) {
  return (unsigned long long)(v + (1LL << 59)) > (2ULL << 59);
}

// Block sum of doubles and of (hi, lo) integers into one partial per CTA.
template <int NT>
__device__ __forceinline__ void block_sums(double v, long long s, bool sums, double* norm,
                                           long long* psum) {
  constexpr int NW = (NT + 31) / 32;
  __shared__ double wd[NW];
  __shared__ long long wh[NW], wl[NW];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned mask = w == NT / 32 ? (1u << (NT & 31)) - 1 : 0xffffffffu;  // a partial last warp
  long long hi = s >> 32, lo = s & 0xffffffffLL;
  for (int o = 16; o > 0; o >>= 1) {
    const double d = __shfl_down_sync(mask, v, o);
    const long long h = __shfl_down_sync(mask, hi, o), l = __shfl_down_sync(mask, lo, o);
    const bool in = lane + o < 32 && (int)threadIdx.x + o < NT;
    v += in ? d : 0.0;
    hi += in ? h : 0;
    lo += in ? l : 0;
  }
  if (lane == 0) {
    wd[w] = v;
    wh[w] = hi;
    wl[w] = lo;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    long long th = 0, tl = 0;
    for (int q = 0; q < NW; ++q) {
      t += wd[q];
      th += wh[q];
      tl += wl[q];
    }
    const size_t b = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    norm[b] = t;
    if (sums) {
      psum[2 * b] = th;
      psum[2 * b + 1] = tl;
    }
  }
}

// Plane q of the level for a march that may leave it: wrapped, or -1 outside a wall.
__device__ __forceinline__ int plane_of(int q, int nz, bool pz) {
  if (q >= 0 && q < nz) return q;
  return pz ? (q + 2 * nz) % nz : -1;
}

// ---------------------------------------------------------------------------
// Down leg: u_out = SMOOTH(u_in), fc = -(sum of R over the eight children) / 8
// (the restricted defect times h^2 2^S).  Step q: plane q arrives; [A] red
// half-step of plane q - 1; [B] black half-step of q - 2, which is then final
// and written, its black defects from the half-step's own R (the red
// neighbours do not change again: R - 6 delta, and each ghost moves with the
// cell); [C] red defects of q - 3.
template <bool WALLS>
__global__ void __launch_bounds__(Down::NT, 1) k_fx64_down(const __grid_constant__ Fx64Args a) {
  using W = Down;
  extern __shared__ longlong2 fx64_smem[];
  auto& ring = *reinterpret_cast<Ring::Of<W::NT>*>(fx64_smem);
  long long* base = reinterpret_cast<long long*>(fx64_smem + 2 * kRing * W::NT);
  const int t = threadIdx.x;
  const Pair p = make_pair_of<W, 4, 3>(a, t);
  // planes by colour and plane parity: raw black, red after [A], black after
  // [B]; then the odd rows' block sums
  long long* const raw = base + W::PAD + t;
  long long* const red = raw + 2 * W::PLANE;
  long long* const blk = red + 2 * W::PLANE;
  long long* const odd = blk + 2 * W::PLANE;
  const bool pz = ((a.fk >> 8) & 3) == BC_PERIODIC;
  const int nz = a.g.nz, z0 = (int)blockIdx.z * a.cz, z1 = min(z0 + a.cz, nz);
  const unsigned plane = (unsigned)a.g.nx * a.g.ny;
  const unsigned col = (unsigned)p.j * a.g.nx + p.i0;
  auto issue = [&](int q) {
    const int k = q <= z1 + 2 ? plane_of(q, nz, pz) : -1;
    if (k >= 0 && p.valid) {
      const size_t o = (size_t)k * plane + col;
      const int s = (q - z0 + 8) & (kRing - 1);
      cp16(&ring.u[s][t], a.u_in + o);
      cp16(&ring.f[s][t], a.F + o);
    }
    cp_commit();
  };
  // values by plane: P, Q columns of planes a, b, c; what [C] needs of c - 1
  long long uaP = 0, uaQ = 0, ubP = 0, ubQ = 0, ucP = 0, ucQ = 0, ud = 0;
  long long faP = 0, faQ = 0, fbP = 0, fbQ = 0, fcr = 0;
  long long acc = 0, done = 0, psum = 0;
  double norm = 0.0;
  bool bad = false;
  issue(z0 - 3);
  issue(z0 - 2);
  issue(z0 - 1);
  // EVEN: plane q is even
  auto step = [&](auto even, int q) {
    constexpr bool EVEN = decltype(even)::value;
    issue(q + 3);
    cp_wait<3>();
    const int s = (q - z0 + 8) & (kRing - 1);
    longlong2 v = make_longlong2(0, 0), f = v;
    if (p.valid && (!WALLS || plane_of(q, nz, pz) >= 0)) {
      v = ring.u[s][t];
      f = ring.f[s][t];
    }
    const long long uP = p.swap ? v.y : v.x, uQ = p.swap ? v.x : v.y;
    const long long fP = p.swap ? f.y : f.x, fQ = p.swap ? f.x : f.y;
    constexpr int I0 = EVEN ? 0 : W::PLANE, I1 = EVEN ? W::PLANE : 0;  // parity of q, of q - 1
    raw[I0] = EVEN ? uQ : uP;  // P is red in even planes
    if (p.tile && q >= z0 && q < z1) psum += uP + uQ;
    // the block whose last plane was q - 4: its even and odd row's sums
    if (!EVEN && q - 5 >= z0 && q - 5 < z1 && p.tile && !(p.j & 1)) {
      const long long sum = done + odd[W::PW];
      const int K = (q - 5) >> 1;
      a.fc[((size_t)K * (a.g.ny >> 1) + (p.j >> 1)) * (a.g.nx >> 1) + (p.i0 >> 1)] =
          cvt::ll2d_pow2_rn(-sum, 3);
    }
    const int ka = q - 1, kb = q - 2, kc = q - 3;
    // [A] plane q - 1 (the other parity): red is Q there when q is even
    {
      const int wl = WALLS && !pz && ka == 0 ? wall_sign(a.fk, 4) : 0;
      const int wh = WALLS && !pz && ka == nz - 1 ? wall_sign(a.fk, 5) : 0;
      long long& r = EVEN ? uaQ : uaP;
      const long long R =
          sum6<WALLS, W::PW>(raw + I1, r, EVEN ? uaP : uaQ, EVEN ? -p.xo : p.xo,
                             EVEN ? p.wxq : p.wxp, p, EVEN ? ubQ : ubP, EVEN ? uQ : uP, wl, wh) -
          6 * r - (EVEN ? faQ : faP);
      if (p.tile && ka >= z0 && ka < z1) {
        const double d = __ll2double_rn(R);
        norm = fma(d, d, norm);
      }
      r += weigh(R, a.w);
      red[I1] = r;
    }
    // [B] plane q - 2 (parity of q): black is Q there when q is even
    long long rb;
    {
      const int wl = WALLS && !pz && kb == 0 ? wall_sign(a.fk, 4) : 0;
      const int wh = WALLS && !pz && kb == nz - 1 ? wall_sign(a.fk, 5) : 0;
      long long& b = EVEN ? ubQ : ubP;
      const long long R =
          sum6<WALLS, W::PW>(red + I0, b, EVEN ? ubP : ubQ, EVEN ? -p.xo : p.xo,
                             EVEN ? p.wxq : p.wxp, p, EVEN ? ucQ : ucP, EVEN ? uaQ : uaP, wl, wh) -
          6 * b - (EVEN ? fbQ : fbP);
      const long long d = weigh(R, a.w);
      int n = 6;  // R moves by -d (6 - signs of the ghosts that move with the cell)
      if (WALLS) n -= (EVEN ? p.wxq : p.wxp) + p.wyl + p.wyh + wl + wh;
      b += d;
      rb = R - n * d;
      blk[I0] = b;
      if (p.tile && kb >= z0 && kb < z1) {
        bad |= too_large(ubP) || too_large(ubQ);
        const size_t o = (size_t)kb * plane + col;
        *reinterpret_cast<longlong2*>(a.u_out + o) =
            p.swap ? make_longlong2(ubQ, ubP) : make_longlong2(ubP, ubQ);
      }
    }
    // [C] plane q - 3 (the other parity): red is Q there when q is even
    {
      const int wl = WALLS && !pz && kc == 0 ? wall_sign(a.fk, 4) : 0;
      const int wh = WALLS && !pz && kc == nz - 1 ? wall_sign(a.fk, 5) : 0;
      const long long r = EVEN ? ucQ : ucP;
      const long long R =
          sum6<WALLS, W::PW>(blk + I1, r, EVEN ? ucP : ucQ, EVEN ? -p.xo : p.xo,
                             EVEN ? p.wxq : p.wxp, p, ud, EVEN ? ubQ : ubP, wl, wh) -
          6 * r - fcr;
      // planes kc (odd when q is even) and kb of blocks (2K, 2K + 1)
      if (EVEN) {  // kc closes its block, kb opens the next
        done = acc + R;
        acc = rb;
        if (p.j & 1) *odd = done;
      } else {
        acc += R + rb;
      }
    }
    // the next plane's [C] needs the black of this q - 3 in the column of its red
    ud = EVEN ? ucP : ucQ;
    ucP = ubP;
    ucQ = ubQ;
    fcr = EVEN ? fbP : fbQ;
    ubP = uaP;
    ubQ = uaQ;
    fbP = faP;
    fbQ = faQ;
    uaP = uP;
    uaQ = uQ;
    faP = fP;
    faQ = fQ;
    __syncthreads();
  };
  // z0 is even, so the march starts on an odd plane
  for (int q = z0 - 3; q <= z1 + 3; q += 2) {
    step(std::false_type{}, q);
    step(std::true_type{}, q + 1);
  }
  cp_wait<0>();
  if (bad) atomicOr(a.flag, 1);
  block_sums<W::NT>(norm, psum, true, a.norm, a.psum);
}

// ---------------------------------------------------------------------------
// Up leg: u_out = SMOOTH(u_in + trilinear(ec)).  Step q: plane q arrives and
// gets its correction; [A] red half-step of q - 1; [B] black half-step of
// q - 2, then final and written.  The correction of a pair is interpolated
// along y, then x, then z with weights 3 and 1 on the integer grid and rounded
// once by the division by 64.
template <bool WALLS>
__global__ void __launch_bounds__(Up::NT, 1) k_fx64_up(const __grid_constant__ Fx64Args a) {
  using W = Up;
  extern __shared__ longlong2 fx64_smem[];
  auto& ring = *reinterpret_cast<Ring::Of<W::NT>*>(fx64_smem);
  long long* base = reinterpret_cast<long long*>(fx64_smem + 2 * kRing * W::NT);
  const int t = threadIdx.x;
  const Pair p = make_pair_of<W, 2, 2>(a, t);
  long long* const raw = base + W::PAD + t;
  long long* const red = raw + 2 * W::PLANE;
  const bool pz = ((a.fk >> 8) & 3) == BC_PERIODIC;
  const int nz = a.g.nz, z0 = (int)blockIdx.z * a.cz, z1 = min(z0 + a.cz, nz);
  const unsigned plane = (unsigned)a.g.nx * a.g.ny;
  const unsigned col = (unsigned)p.j * a.g.nx + p.i0;
  auto issue = [&](int q) {
    const int k = q <= z1 + 1 ? plane_of(q, nz, pz) : -1;
    if (k >= 0 && p.valid) {
      const size_t o = (size_t)k * plane + col;
      const int s = (q - z0 + 8) & (kRing - 1);
      cp16(&ring.u[s][t], a.u_in + o);
      cp16(&ring.f[s][t], a.F + o);
    }
    cp_commit();
  };
  // coarse columns m - 1, m, m + 1 of rows J and J': offsets and signs
  const int nxc = a.g.nx >> 1, nyc = a.g.ny >> 1, nzc = nz >> 1, m = p.i0 >> 1, J = p.j >> 1;
  int ml = m - 1, mh = m + 1, J2 = (p.j & 1) ? J + 1 : J - 1, sl = 1, sh = 1, sy = 1;
  if (ml < 0) {
    const int s = wall_sign(a.fk, 0);
    ml = s ? 0 : nxc - 1;
    sl = s ? s : 1;
  }
  if (mh >= nxc) {
    const int s = wall_sign(a.fk, 1);
    mh = s ? nxc - 1 : 0;
    sh = s ? s : 1;
  }
  if (J2 < 0 || J2 >= nyc) {
    const int lo = J2 < 0, s = wall_sign(a.fk, lo ? 2 : 3);
    J2 = lo == (s == 0) ? nyc - 1 : 0;
    sy = s ? s : 1;
  }
  const unsigned planec = (unsigned)nxc * nyc;
  const unsigned r1 = (unsigned)J * nxc, r2 = (unsigned)J2 * nxc;
  long long c1[3], c2[3];  // the next coarse plane's values, loaded ahead
  int sz = 1;
  auto load_coarse = [&](int K) {
    int Kw = K;
    sz = 1;
    if (K < 0 || K >= nzc) {
      const int lo = K < 0, s = wall_sign(a.fk, lo ? 4 : 5);
      Kw = s ? (lo ? 0 : nzc - 1) : (K + 2 * nzc) % nzc;
      sz = s ? s : 1;
    }
    const long long* e = a.ec + (size_t)Kw * planec;
    c1[0] = e[r1 + ml];
    c1[1] = e[r1 + m];
    c1[2] = e[r1 + mh];
    c2[0] = e[r2 + ml];
    c2[1] = e[r2 + m];
    c2[2] = e[r2 + mh];
  };
  // 16 times the (x, y) interpolation of the loaded plane at the pair's cells
  auto interp = [&](long long& v0, long long& v1) {
    long long w[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) w[x] = 3 * c1[x] + (WALLS ? signed_by(sy, c2[x]) : c2[x]);
    if (WALLS) {
      w[0] = signed_by(sl, w[0]);
      w[2] = signed_by(sh, w[2]);
    }
    v0 = 3 * w[1] + w[0];
    v1 = 3 * w[1] + w[2];
    if (WALLS) {
      v0 = signed_by(sz, v0);
      v1 = signed_by(sz, v1);
    }
  };
  long long em0, em1, e00, e01;  // coarse planes K - 1 and K
  long long uaP = 0, uaQ = 0, ubP = 0, ubQ = 0, uc = 0;
  long long faP = 0, faQ = 0, fbb = 0;
  double norm = 0.0;
  bool bad = false;
  issue(z0 - 2);
  issue(z0 - 1);
  issue(z0);
  load_coarse((z0 >> 1) - 2);
  interp(em0, em1);
  load_coarse((z0 >> 1) - 1);
  interp(e00, e01);
  load_coarse(z0 >> 1);
  auto step = [&](auto even, int q) {
    constexpr bool EVEN = decltype(even)::value;
    issue(q + 3);
    cp_wait<3>();
    const int s = (q - z0 + 8) & (kRing - 1);
    longlong2 v = make_longlong2(0, 0), f = v;
    if (p.valid && (!WALLS || plane_of(q, nz, pz) >= 0)) {
      v = ring.u[s][t];
      f = ring.f[s][t];
    }
    if (EVEN) {  // planes K - 1, K
      v.x += (3 * e00 + em0 + 32) >> 6;
      v.y += (3 * e01 + em1 + 32) >> 6;
    } else {  // planes K, K + 1
      long long p0, p1;
      interp(p0, p1);
      v.x += (3 * e00 + p0 + 32) >> 6;
      v.y += (3 * e01 + p1 + 32) >> 6;
      em0 = e00;
      em1 = e01;
      e00 = p0;
      e01 = p1;
      load_coarse(((q + 1) >> 1) + 1);
    }
    const long long uP = p.swap ? v.y : v.x, uQ = p.swap ? v.x : v.y;
    const long long fP = p.swap ? f.y : f.x, fQ = p.swap ? f.x : f.y;
    constexpr int I0 = EVEN ? 0 : W::PLANE, I1 = EVEN ? W::PLANE : 0;
    raw[I0] = EVEN ? uQ : uP;
    const int ka = q - 1, kb = q - 2;
    {
      const int wl = WALLS && !pz && ka == 0 ? wall_sign(a.fk, 4) : 0;
      const int wh = WALLS && !pz && ka == nz - 1 ? wall_sign(a.fk, 5) : 0;
      long long& r = EVEN ? uaQ : uaP;
      const long long R =
          sum6<WALLS, W::PW>(raw + I1, r, EVEN ? uaP : uaQ, EVEN ? -p.xo : p.xo,
                             EVEN ? p.wxq : p.wxp, p, EVEN ? ubQ : ubP, EVEN ? uQ : uP, wl, wh) -
          6 * r - (EVEN ? faQ : faP);
      r += weigh(R, a.w);
      red[I1] = r;
    }
    {
      const int wl = WALLS && !pz && kb == 0 ? wall_sign(a.fk, 4) : 0;
      const int wh = WALLS && !pz && kb == nz - 1 ? wall_sign(a.fk, 5) : 0;
      long long& b = EVEN ? ubQ : ubP;
      const long long R =
          sum6<WALLS, W::PW>(red + I0, b, EVEN ? ubP : ubQ, EVEN ? -p.xo : p.xo,
                             EVEN ? p.wxq : p.wxp, p, uc, EVEN ? uaQ : uaP, wl, wh) -
          6 * b - fbb;
      const long long d = weigh(R, a.w);
      int n = 6;
      if (WALLS) n -= (EVEN ? p.wxq : p.wxp) + p.wyl + p.wyh + wl + wh;
      b += d;
      if (p.tile && kb >= z0 && kb < z1) {
        bad |= too_large(ubP) || too_large(ubQ);
        const double x = __ll2double_rn(R - n * d);
        norm = fma(x, x, norm);
        const size_t o = (size_t)kb * plane + col;
        *reinterpret_cast<longlong2*>(a.u_out + o) =
            p.swap ? make_longlong2(ubQ, ubP) : make_longlong2(ubP, ubQ);
      }
    }
    // the next plane's [B] needs the red of this q - 2 in the column of its
    // black, and the F of its black
    uc = EVEN ? ubP : ubQ;
    fbb = EVEN ? faP : faQ;
    ubP = uaP;
    ubQ = uaQ;
    uaP = uP;
    uaQ = uQ;
    faP = fP;
    faQ = fQ;
    __syncthreads();
  };
  // z0 is even: the march starts on an even plane
  for (int q = z0 - 2; q <= z1; q += 2) {
    step(std::true_type{}, q);
    step(std::false_type{}, q + 1);
  }
  cp_wait<0>();
  if (bad) atomicOr(a.flag, 1);
  block_sums<W::NT>(norm, 0, false, a.norm, nullptr);
}

template <typename W>
constexpr size_t smem_bytes(int planes) {
  return sizeof(Ring::Of<W::NT>) + (size_t)planes * W::PLANE * sizeof(long long);
}
constexpr size_t kDownSmem = smem_bytes<Down>(7), kUpSmem = smem_bytes<Up>(4);

// In place: f becomes F = round(f c) - sum over the cell's fixed and open
// faces of round(2 b 2^S) (c2 = 2^(S+1)).
__global__ void k_fx64_source(double* f, Grid g, Bc bc, double c, double c2) {
  long long* q = reinterpret_cast<long long*>(f);
  const dev::Split sp(g.nx, g.ny);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < g.cells();
       t += (long long)gridDim.x * blockDim.x) {
    int i, j, k;
    sp(t, i, j, k);
    long long v = cvt::d2ll_rn(f[t] * c);
    if (i == 0 || i == g.nx - 1 || j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1) {
      for (int s = 0; s < 6; ++s) {
        const int kind = face_kind(bc, s);
        if (kind != BC_FIXED && kind != BC_OPEN) continue;
        const int x = s < 2 ? i : s < 4 ? j : k, n = s < 2 ? g.nx : s < 4 ? g.ny : g.nz;
        if (x != ((s & 1) ? n - 1 : 0)) continue;
        v -= __double2ll_rn(dev::face_value(bc, g, s, (s < 2 ? j : i) + 1, (s < 4 ? k : j) + 1) *
                            c2);
      }
    }
    q[t] = v;
  }
}

// out[0] = sum of a[0 .. n) + sum of b[0 .. nb), in a fixed order.
__global__ void k_fx64_norm(const double* a, int n, const double* b, int nb, double* out) {
  __shared__ double ws[8];
  double s = 0.0;
  for (int t = threadIdx.x; t < n; t += blockDim.x) s += a[t];
  for (int t = threadIdx.x; t < nb; t += blockDim.x) s += b[t];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int w = 0; w < 8; ++w) r += ws[w];
    out[0] = r;
  }
}

Weight weight_of(double omega) {
  const double x = std::ldexp(omega / 6.0, 32), hi = std::nearbyint(x);  // x - hi is exact
  const double lo = std::nearbyint(std::ldexp(x - hi, 32));
  return Weight{(int)hi, lo >= 2147483647.0 ? 2147483647 : (int)lo};
}

cudaError_t configure() {
  static std::atomic<int> configured[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && configured[dev].load()) return cudaSuccess;
  struct {
    const void* f;
    size_t b;
  } k[4] = {{(const void*)k_fx64_down<false>, kDownSmem},
            {(const void*)k_fx64_down<true>, kDownSmem},
            {(const void*)k_fx64_up<false>, kUpSmem},
            {(const void*)k_fx64_up<true>, kUpSmem}};
  for (auto& x : k) {
    const cudaError_t e =
        cudaFuncSetAttribute(x.f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)x.b);
    if (e != cudaSuccess) return e;
  }
  if (dev >= 0 && dev < 64) configured[dev].store(1);
  return cudaSuccess;
}

}  // namespace

bool fx64_ok(Grid g) {
  return g.nx % TX == 0 && g.ny % TY == 0 && g.nz % 2 == 0 && g.nz >= 16 &&
         g.cells() <= (1LL << 30) && fx64_blocks(g) <= kPartials;
}

// Planes per CTA: the even count for which the last wave of CTAs (one per SM)
// is best filled, counting the six planes a chunk's halo costs; at most 128 (a
// thread's exact sum of its columns' integers must stay below 2^63).
int fx64_cz(Grid g) {
  const long long cols = (long long)(g.nx / TX) * (g.ny / TY);
  int best = 0;
  long long least = 0;
  for (int cz = 4; cz <= 128 && cz <= g.nz; cz += 2) {
    const long long ctas = cols * ((g.nz + cz - 1) / cz);
    if (ctas > kPartials) continue;
    const long long cost = (ctas + sm_count() - 1) / sm_count() * (cz + 6);
    if (best == 0 || cost < least) {
      best = cz;
      least = cost;
    }
  }
  return best;
}

int fx64_blocks(Grid g) {
  const int cz = fx64_cz(g);
  if (cz == 0) return 1 << 30;
  return (int)((long long)(g.nx / TX) * (g.ny / TY) * ((g.nz + cz - 1) / cz));
}

static int face_kinds_of(const Bc& hom) {
  int fk = 0;
  for (int q = 0; q < 6; ++q) fk |= face_kind(hom, q) << (2 * q);
  return fk;
}

cudaError_t launch_fx64_down(const long long* u_in, long long* u_out, const long long* F, double* fc,
                             Grid g, const Bc& hom, double omega, double* norm, long long* psum,
                             int* flag, cudaStream_t s) {
  const cudaError_t e = configure();
  if (e != cudaSuccess) return e;
  Fx64Args a{};
  a.u_in = u_in;
  a.u_out = u_out;
  a.F = F;
  a.g = g;
  a.fk = face_kinds_of(hom);
  a.cz = fx64_cz(g);
  a.w = weight_of(omega);
  a.norm = norm;
  a.fc = fc;
  a.psum = psum;
  a.flag = flag;
  const dim3 grid(g.nx / TX, g.ny / TY, (g.nz + a.cz - 1) / a.cz);
  ++g_launches;
  if (a.fk) k_fx64_down<true><<<grid, Down::NT, kDownSmem, s>>>(a);
  else k_fx64_down<false><<<grid, Down::NT, kDownSmem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_fx64_up(const long long* u_in, long long* u_out, const long long* F,
                           const long long* ec, Grid g, const Bc& hom, double omega, double* norm,
                           int* flag, cudaStream_t s) {
  const cudaError_t e = configure();
  if (e != cudaSuccess) return e;
  Fx64Args a{};
  a.u_in = u_in;
  a.u_out = u_out;
  a.F = F;
  a.g = g;
  a.fk = face_kinds_of(hom);
  a.cz = fx64_cz(g);
  a.w = weight_of(omega);
  a.norm = norm;
  a.ec = ec;
  a.flag = flag;
  const dim3 grid(g.nx / TX, g.ny / TY, (g.nz + a.cz - 1) / a.cz);
  ++g_launches;
  if (a.fk) k_fx64_up<true><<<grid, Up::NT, kUpSmem, s>>>(a);
  else k_fx64_up<false><<<grid, Up::NT, kUpSmem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_fx64_source(double* f, Grid g, const Bc& bc, double c, double two_pow_S,
                               cudaStream_t s) {
  long long b = (g.cells() + 255) / 256;
  if (b > sm_count() * 64LL) b = sm_count() * 64LL;
  ++g_launches;
  k_fx64_source<<<(int)b, 256, 0, s>>>(f, g, bc, c, 2.0 * two_pow_S);
  return cudaGetLastError();
}

cudaError_t launch_fx64_norm(const double* red, const double* black, int nb, double* out,
                             cudaStream_t s) {
  ++g_launches;
  k_fx64_norm<<<1, 256, 0, s>>>(red, nb, black, nb, out);
  return cudaGetLastError();
}

}  // namespace mg
