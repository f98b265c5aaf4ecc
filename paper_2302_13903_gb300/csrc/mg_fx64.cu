// mg_fx64.cu -- the levels of the FP64 path from 64^3 up in exact 64-bit fixed
// point.
//
// An SM issues two FP64 operations per clock, so a V(1,1) cycle's 25-30 FP64
// operations per cell take several times as long as its bytes.  Here phi and
// h^2 f of the finest level are 64-bit integers scaled by 2^S, S so large that
// twice the largest |phi| of the FMG start on the next level lies between 2^56
// and 2^57 (or h^2 max|f| between 2^57 and 2^58): a quantum of 2^-56 to 2^-55
// of max|phi|, an eighth to a quarter of the spacing of doubles there.  Cells
// more than that below max|phi| have fewer bits than doubles have; every cell's
// update carries an eighth of the rounding that an FP64 update carries where |phi| is
// largest.  With U and F those integers,
//   R = (sum of the six neighbours of U) - 6 U - F       (exactly)
//   SMOOTH: U += round(R omega / 6)                      (Eqs. rbsor1-rbsor2)
//   defect: f - L u = -R / (h^2 2^S)                     (Eq. defect)
// so neighbour sums and defects carry no rounding at all, and one update rounds
// once.  omega / 6 is a 64-bit fraction.  A face's value b enters the ghost 2 b - u as a
// constant and is folded into F (F - round(2 b 2^S)) when F is formed, so the
// sweeps run the homogeneous rule.
//
// The levels below, down to 64^3, hold the correction on the same grid: with h_c
// = 2 h their right-hand side is F_c = -(sum of R) / 2, so no scale has to be
// found, and a correction has the quantum of the phi it is added to.
//
// Ranges: |U| < 2^59 on the finest level and |F| < 2^60 keep |R| below 2^63; the
// flag is raised where a U passes that, a correction 2^56 (its interpolation has
// weights of 64 in all) or a coarse F 2^60, and the solve then runs in FP64.  The
// sum of R over eight cells is not checked on its own: past 2^63 it is one wrong
// correction, which the next norm, exact always, shows.
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
#include <type_traits>

#include "mg_convert.cuh"
#include "mg_device.cuh"
#include "mg_internal.h"
#include "mg_sums.h"

namespace mg {
namespace {

constexpr int TY = 16;
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
  double* fc;           // down: coarse right-hand side, -sum of R, as doubles,
  long long* fci;       //   or half of it, as F of an integer level (fc null)
  const long long* ec;  // up: coarse correction on the integer grid
  int limit;            // log2 of the largest |U|
  int* flag;            // |U| or |F| of the coarse level passed its limit
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
__device__ __forceinline__ void cp8(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// The pairs of a CTA: its TX x TY tile and a halo of HX cells and HY rows.
template <int TX_, int HX_, int HY_>
struct Win {
  static constexpr int TX = TX_, HX = HX_, HY = HY_;
  static constexpr int PW = (TX + 2 * HX) / 2;  // pairs per row
  static constexpr int RH = TY + 2 * HY;
  static constexpr int NT = PW * RH;
  static constexpr int PAD = PW + 1;  // so that every neighbour index is in range
  static constexpr int PLANE = NT + 2 * PAD;
};
// The down leg reads the raw black cells of one more row on either side: the
// first 2 PW threads bring those in, so that no thread computes them.
template <int TX>
using Down = Win<TX, 4, 2>;
template <int TX>
using Up = Win<TX, 2, 2>;

template <int NT, int NF>
struct Ring {
  longlong2 u[kRing][NT];
  longlong2 f[kRing][NT];
  long long frame[kRing][NF];
};

// What a thread knows about its pair of columns.  Column P is the one that is
// red in even planes, column Q the one that is red in odd planes.
struct Pair {
  int i0, j;   // cells (i0, j) and (i0 + 1, j), wrapped into the level
  bool valid;  // inside the level
  bool tile;   // written by this CTA
  bool swap;   // P is cell i0 + 1
  int xo;      // pair offset of P's neighbour outside the pair (Q's is -xo)
  int n;       // 6 less the signs of the ghosts across x and y walls of P, of Q << 8
};

__device__ __forceinline__ int wall_sign(int fk, int q) {
  const int kind = (fk >> (2 * q)) & 3;
  return kind == BC_PERIODIC ? 0 : kind == BC_ZEROGRAD ? 1 : -1;
}

template <typename W>
__device__ __forceinline__ Pair make_pair_of(const Fx64Args& a, int pm, int pr) {
  Pair p;
  int i = (int)blockIdx.x * W::TX + 2 * pm - W::HX, j = (int)blockIdx.y * TY + pr - W::HY;
  p.tile = pm >= W::HX / 2 && pm < (W::HX + W::TX) / 2 && pr >= W::HY && pr < W::HY + TY;
  const bool px = (a.fk & 3) == BC_PERIODIC, py = ((a.fk >> 4) & 3) == BC_PERIODIC;
  p.valid = (px || (i >= 0 && i < a.g.nx)) && (py || (j >= 0 && j < a.g.ny));
  p.swap = j & 1;
  p.xo = p.swap ? 1 : -1;
  const int xl = i == 0 ? wall_sign(a.fk, 0) : 0, xh = i + 2 == a.g.nx ? wall_sign(a.fk, 1) : 0;
  const int y = j == 0 ? wall_sign(a.fk, 2) : j == a.g.ny - 1 ? wall_sign(a.fk, 3) : 0;
  p.n = (6 - (p.swap ? xh : xl) - y) | (6 - (p.swap ? xl : xh) - y) << 8;
  i = i < 0 ? i + a.g.nx : i >= a.g.nx ? i - a.g.nx : i;
  j = j < 0 ? j + a.g.ny : j >= a.g.ny ? j - a.g.ny : j;
  p.i0 = p.valid ? i : 0;
  p.j = p.valid ? j : 0;
  return p;
}

__device__ __forceinline__ long long signed_by(int s, long long v) { return s < 0 ? -v : v; }

// (Sum of the six neighbours) - 6 self - F of a cell whose neighbours of the
// plane are in o (at this thread's index); `mate` is the pair's other cell, xo
// the offset of the neighbour outside the pair, zl and zh the planes below and
// above.  A ghost across a wall is +-self: cells outside the level hold 0, and
// n is 6 less the ghosts' signs.
template <int PW>
__device__ __forceinline__ long long residual(const long long* o, long long self, long long mate,
                                              int xo, long long zl, long long zh, int n,
                                              long long F) {
  return (((mate + o[xo]) + (o[-PW] + o[PW])) + (zl + zh)) - n * self - F;
}

// |v| at or past 2^32 m, by the high word.
__device__ __forceinline__ bool too_large(long long v, int m) {
  return (unsigned)((int)(v >> 32) + m) >= 2u * m;
}

// Block sum into one partial per CTA.
template <int NT>
__device__ __forceinline__ void block_sum(double v, double* norm) {
  constexpr int NW = (NT + 31) / 32;
  __shared__ double wd[NW];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned mask = w == NT / 32 ? (1u << (NT & 31)) - 1 : 0xffffffffu;  // a partial last warp
  for (int o = 16; o > 0; o >>= 1) {
    const double d = __shfl_down_sync(mask, v, o);
    v += lane + o < 32 && (int)threadIdx.x + o < NT ? d : 0.0;
  }
  if (lane == 0) wd[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < NW; ++q) t += wd[q];
    norm[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
  }
}

// Plane q of the level (-nz <= q < 2 nz) for a march that may leave it:
// wrapped, or -1 outside a wall.
__device__ __forceinline__ int plane_of(int q, int nz, bool pz) {
  const int k = q < 0 ? q + nz : q >= nz ? q - nz : q;
  return pz || k == q ? k : -1;
}

// ---------------------------------------------------------------------------
// Down leg: u_out = SMOOTH(u_in), fc = -(sum of R over the eight children) (8
// times the restricted defect times h^2 2^S).  Step q: plane q arrives; [A] red
// half-step of plane q - 1; [B] black half-step of q - 2, which is then final
// and written, its black defects from the half-step's own R (the red
// neighbours do not change again: R - 6 delta, and each ghost moves with the
// cell); [C] red defects of q - 3.  The march is unrolled by four, so that ring
// slots and the registers of the four planes in hand are fixed: plane q is in
// slot J, planes q - 1, q - 2, q - 3 in J - 1, J - 2, J - 3 (mod 4).
// COARSE: a correction level, from u = 0 and without the norm.
template <bool WALLS, int TX, bool COARSE>
__global__ void __launch_bounds__(Down<TX>::NT)
    k_fx64_down(const __grid_constant__ Fx64Args a) {
  dev::after_previous();
  using W = Down<TX>;
  extern __shared__ longlong2 fx64_smem[];
  using R = Ring<W::NT, 2 * W::PW>;
  R& ring = *reinterpret_cast<R*>(fx64_smem);
  long long* base = reinterpret_cast<long long*>(&ring + 1);
  const int t = threadIdx.x;
  const Pair p = make_pair_of<W>(a, t % W::PW, t / W::PW);
  // planes by colour and plane parity: raw black, red after [A], black after
  // [B]; then the odd rows' block sums
  long long* const raw = base + W::PAD + t;
  long long* const red = raw + 2 * W::PLANE;
  long long* const blk = red + 2 * W::PLANE;
  long long* const odd = blk + 2 * W::PLANE;
  const bool pz = ((a.fk >> 8) & 3) == BC_PERIODIC;
  const int wzl = WALLS ? wall_sign(a.fk, 4) : 0, wzh = WALLS ? wall_sign(a.fk, 5) : 0;
  const int nz = a.g.nz, z0 = (int)blockIdx.z * a.cz, z1 = min(z0 + a.cz, nz);
  const unsigned plane = (unsigned)a.g.nx * a.g.ny;
  const unsigned col = (unsigned)p.j * a.g.nx + p.i0;
  const unsigned colc = (unsigned)(p.j >> 1) * (a.g.nx >> 1) + (p.i0 >> 1);
  const bool even_row = p.tile && !(p.j & 1), odd_row = p.j & 1;
  // the frame: column of Q (black in even planes) and its distance to P's
  const bool framed = t < 2 * W::PW;
  const Pair fp = make_pair_of<W>(a, t % W::PW, t < W::PW ? -1 : W::RH);
  const bool frame_in = framed && fp.valid;
  const unsigned fcol = (unsigned)fp.j * a.g.nx + fp.i0 + (fp.swap ? 0 : 1);
  const int fstep = fp.swap ? 1 : -1;
  long long* const frame = raw + (t < W::PW ? -W::PW : W::NT - W::PW);
  auto issue = [&](auto slot, int q) {
    constexpr int s = decltype(slot)::value & 3;
    const int k = q <= z1 + 2 ? plane_of(q, nz, pz) : -1;
    if (k >= 0 && (!WALLS || p.valid)) {
      const size_t o = (size_t)k * plane + col;
      if (!COARSE) cp16(&ring.u[s][t], a.u_in + o);
      cp16(&ring.f[s][t], a.F + o);
    }
    if (!COARSE && k >= 0 && frame_in)  // odd slots hold even planes
      cp8(&ring.frame[s][t], a.u_in + (size_t)k * plane + fcol + (s & 1 ? 0 : fstep));
    cp_commit();
  };
  long long uP[4] = {}, uQ[4] = {}, fP[4] = {}, fQ[4] = {};
  long long ud = 0, acc = 0, done = 0;
  // outside the level cells stay 0
  auto delta = [&](long long R) { return !WALLS || p.valid ? weigh(R, a.w) : 0; };
  const int most = 1 << (a.limit - 32);
  SquareSum norm;
  bool bad = false;
  using std::integral_constant;
  issue(integral_constant<int, 0>{}, z0 - 3);
  issue(integral_constant<int, 1>{}, z0 - 2);
  issue(integral_constant<int, 2>{}, z0 - 1);
  auto step = [&](auto Jc, int q) {
    constexpr int J = decltype(Jc)::value, A = (J + 3) & 3, B = (J + 2) & 3, C = (J + 1) & 3;
    constexpr bool EVEN = J & 1;  // q is even (the march starts on an odd plane)
    constexpr int I0 = EVEN ? 0 : W::PLANE, I1 = EVEN ? W::PLANE : 0;  // parity of q, of q - 1
    // the columns by what they are in planes of q's parity; in planes of the
    // other parity red and black change places
    long long(&uR)[4] = EVEN ? uP : uQ;
    long long(&uB)[4] = EVEN ? uQ : uP;
    long long(&fR)[4] = EVEN ? fP : fQ;
    long long(&fB)[4] = EVEN ? fQ : fP;
    const int xb = EVEN ? -p.xo : p.xo, nb = WALLS ? (EVEN ? p.n >> 8 : p.n & 255) : 6;
    issue(integral_constant<int, J + 3>{}, q + 3);
    cp_wait<3>();
    if (!WALLS || p.valid) {
      const longlong2 v = COARSE ? make_longlong2(0, 0) : ring.u[J][t], f = ring.f[J][t];
      uP[J] = p.swap ? v.y : v.x;
      uQ[J] = p.swap ? v.x : v.y;
      fP[J] = p.swap ? f.y : f.x;
      fQ[J] = p.swap ? f.x : f.y;
    }
    if (!COARSE) {
      raw[I0] = uB[J];
      if (framed) frame[I0] = frame_in ? ring.frame[J][t] : 0;
    }
    // the block whose last plane was q - 4: its even and odd row's sums
    if (!EVEN && q - 5 >= z0 && q - 5 < z1 && even_row) {
      const long long sum = -(done + odd[W::PW]);
      const size_t o = (size_t)((q - 5) >> 1) * (plane >> 2) + colc;
      if (a.fci) {
        const long long f = (sum + ((sum >> 1) & 1)) >> 1;  // ties to even: no bias
        a.fci[o] = f;
        bad |= too_large(f, 1 << 28);
      } else {
        a.fc[o] = cvt::ll2d_rn(sum);
      }
    }
    const int ka = q - 1, kb = q - 2, kc = q - 3;
    {  // [A]: red of plane q - 1 is in the columns uB
      long long zl = uB[B], zh = uB[J];
      int n = nb;
      if (WALLS && wzl && ka == 0) zl = 0, n -= wzl;
      if (WALLS && wzh && ka == nz - 1) zh = 0, n -= wzh;
      const long long R =
          COARSE ? -fB[A] : residual<W::PW>(raw + I1, uB[A], uR[A], xb, zl, zh, n, fB[A]);
      if (!COARSE && p.tile && ka >= z0 && ka < z1) norm.add(R);
      uB[A] += delta(R);
      red[I1] = uB[A];
    }
    long long rb;
    {  // [B]: black of plane q - 2 is in the columns uB
      long long zl = uB[C], zh = uB[A];
      int n = nb;  // R moves by -n d: the ghosts move with the cell
      if (WALLS && wzl && kb == 0) zl = 0, n -= wzl;
      if (WALLS && wzh && kb == nz - 1) zh = 0, n -= wzh;
      const long long R = residual<W::PW>(red + I0, uB[B], uR[B], xb, zl, zh, n, fB[B]);
      const long long d = delta(R);
      uB[B] += d;
      rb = R - n * d;
      blk[I0] = uB[B];
      if (p.tile && kb >= z0 && kb < z1) {
        bad |= too_large(uP[B], most) || too_large(uQ[B], most);
        *reinterpret_cast<longlong2*>(a.u_out + (size_t)kb * plane + col) =
            p.swap ? make_longlong2(uQ[B], uP[B]) : make_longlong2(uP[B], uQ[B]);
      }
    }
    {  // [C]: red of plane q - 3 is in the columns uB
      long long zl = ud, zh = uB[B];
      int n = nb;
      if (WALLS && wzl && kc == 0) zl = 0, n -= wzl;
      if (WALLS && wzh && kc == nz - 1) zh = 0, n -= wzh;
      const long long R = residual<W::PW>(blk + I1, uB[C], uR[C], xb, zl, zh, n, fB[C]);
      // planes kc and kb of the blocks (2K, 2K + 1)
      if (EVEN) {  // kc is odd and closes its block, kb opens the next
        done = acc + R;
        acc = rb;
        if (odd_row) *odd = done;
      } else {
        acc += R + rb;
      }
    }
    ud = uR[C];  // the next plane's [C] has its red in the other column
    __syncthreads();
  };
  for (int q = z0 - 3; q <= z1 + 3; q += 4) {
    step(integral_constant<int, 0>{}, q);
    step(integral_constant<int, 1>{}, q + 1);
    step(integral_constant<int, 2>{}, q + 2);
    step(integral_constant<int, 3>{}, q + 3);
  }
  cp_wait<0>();
  if (bad) atomicOr(a.flag, 1);
  if (!COARSE) block_sum<W::NT>(norm.total(), a.norm);
}

// ---------------------------------------------------------------------------
// Up leg: u_out = SMOOTH(u_in + trilinear(ec)).  Step q: plane q arrives and
// gets its correction; [A] red half-step of q - 1; [B] black half-step of
// q - 2, then final and written.  The correction of a pair is interpolated
// along y, then x, then z with weights 3 and 1 on the integer grid and rounded
// once by the division by 64.  Unrolled by four as the down leg.
template <bool WALLS, int TX, bool COARSE>
__global__ void __launch_bounds__(Up<TX>::NT)
    k_fx64_up(const __grid_constant__ Fx64Args a) {
  dev::after_previous();
  using W = Up<TX>;
  extern __shared__ longlong2 fx64_smem[];
  using R = Ring<W::NT, 1>;
  R& ring = *reinterpret_cast<R*>(fx64_smem);
  long long* base = reinterpret_cast<long long*>(&ring + 1);
  const int t = threadIdx.x;
  const Pair p = make_pair_of<W>(a, t % W::PW, t / W::PW);
  long long* const raw = base + W::PAD + t;
  long long* const red = raw + 2 * W::PLANE;
  const bool pz = ((a.fk >> 8) & 3) == BC_PERIODIC;
  const int wzl = WALLS ? wall_sign(a.fk, 4) : 0, wzh = WALLS ? wall_sign(a.fk, 5) : 0;
  const int nz = a.g.nz, z0 = (int)blockIdx.z * a.cz, z1 = min(z0 + a.cz, nz);
  const unsigned plane = (unsigned)a.g.nx * a.g.ny;
  const unsigned col = (unsigned)p.j * a.g.nx + p.i0;
  auto issue = [&](auto slot, int q) {
    constexpr int s = decltype(slot)::value & 3;
    const int k = q <= z1 + 1 ? plane_of(q, nz, pz) : -1;
    if (k >= 0 && (!WALLS || p.valid)) {
      const size_t o = (size_t)k * plane + col;
      cp16(&ring.u[s][t], a.u_in + o);
      cp16(&ring.f[s][t], a.F + o);
    }
    cp_commit();
  };
  // coarse columns m - 1, m, m + 1 of rows J and J': offsets and signs
  const int nxc = a.g.nx >> 1, nyc = a.g.ny >> 1, nzc = nz >> 1, m = p.i0 >> 1, J1 = p.j >> 1;
  int ml = m - 1, mh = m + 1, J2 = (p.j & 1) ? J1 + 1 : J1 - 1, sl = 1, sh = 1, sy = 1, sz = 1;
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
  const unsigned r1 = (unsigned)J1 * nxc, r2 = (unsigned)J2 * nxc;
  long long c1[3], c2[3];  // the next coarse plane's values, loaded ahead
  auto load_coarse = [&](int K) {
    int Kw = K;
    sz = 1;
    if (K < 0 || K >= nzc) {
      const int lo = K < 0, s = wall_sign(a.fk, lo ? 4 : 5);
      Kw = s ? (lo ? 0 : nzc - 1) : lo ? K + nzc : K - nzc;
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
  long long uP[4] = {}, uQ[4] = {}, fP[4] = {}, fQ[4] = {};
  // outside the level cells stay 0
  auto delta = [&](long long R) { return !WALLS || p.valid ? weigh(R, a.w) : 0; };
  const int most = 1 << (a.limit - 32);
  SquareSum norm;
  bool bad = false;
  using std::integral_constant;
  issue(integral_constant<int, 0>{}, z0 - 2);
  issue(integral_constant<int, 1>{}, z0 - 1);
  issue(integral_constant<int, 2>{}, z0);
  load_coarse((z0 >> 1) - 2);
  interp(em0, em1);
  load_coarse((z0 >> 1) - 1);
  interp(e00, e01);
  load_coarse(z0 >> 1);
  auto step = [&](auto Jc, int q) {
    constexpr int J = decltype(Jc)::value, A = (J + 3) & 3, B = (J + 2) & 3, C = (J + 1) & 3;
    constexpr bool EVEN = !(J & 1);  // q is even (the march starts on an even plane)
    constexpr int I0 = EVEN ? 0 : W::PLANE, I1 = EVEN ? W::PLANE : 0;
    long long(&uR)[4] = EVEN ? uP : uQ;
    long long(&uB)[4] = EVEN ? uQ : uP;
    long long(&fB)[4] = EVEN ? fQ : fP;
    const int xb = EVEN ? -p.xo : p.xo, nb = WALLS ? (EVEN ? p.n >> 8 : p.n & 255) : 6;
    issue(integral_constant<int, J + 3>{}, q + 3);
    cp_wait<3>();
    long long d0, d1;  // the pair's correction
    if (EVEN) {        // planes K - 1, K
      d0 = 3 * e00 + em0;
      d1 = 3 * e01 + em1;
    } else {  // planes K, K + 1
      long long p0, p1;
      interp(p0, p1);
      d0 = 3 * e00 + p0;
      d1 = 3 * e01 + p1;
      em0 = e00;
      em1 = e01;
      e00 = p0;
      e01 = p1;
      load_coarse(((q + 1) >> 1) + 1);
    }
    if (!WALLS || p.valid) {
      const longlong2 v = ring.u[J][t], f = ring.f[J][t];
      const long long v0 = v.x + ((d0 + 32) >> 6), v1 = v.y + ((d1 + 32) >> 6);
      uP[J] = p.swap ? v1 : v0;
      uQ[J] = p.swap ? v0 : v1;
      fP[J] = p.swap ? f.y : f.x;
      fQ[J] = p.swap ? f.x : f.y;
    }
    raw[I0] = uB[J];
    const int ka = q - 1, kb = q - 2;
    {  // [A]: red of plane q - 1 is in the columns uB
      long long zl = uB[B], zh = uB[J];
      int n = nb;
      if (WALLS && wzl && ka == 0) zl = 0, n -= wzl;
      if (WALLS && wzh && ka == nz - 1) zh = 0, n -= wzh;
      const long long R = residual<W::PW>(raw + I1, uB[A], uR[A], xb, zl, zh, n, fB[A]);
      uB[A] += delta(R);
      red[I1] = uB[A];
    }
    {  // [B]: black of plane q - 2 is in the columns uB
      long long zl = uB[C], zh = uB[A];
      int n = nb;
      if (WALLS && wzl && kb == 0) zl = 0, n -= wzl;
      if (WALLS && wzh && kb == nz - 1) zh = 0, n -= wzh;
      const long long R = residual<W::PW>(red + I0, uB[B], uR[B], xb, zl, zh, n, fB[B]);
      const long long d = delta(R);
      uB[B] += d;
      if (p.tile && kb >= z0 && kb < z1) {
        if (!COARSE) norm.add(R - n * d);
        bad |= too_large(uP[B], most) || too_large(uQ[B], most);
        *reinterpret_cast<longlong2*>(a.u_out + (size_t)kb * plane + col) =
            p.swap ? make_longlong2(uQ[B], uP[B]) : make_longlong2(uP[B], uQ[B]);
      }
    }
    __syncthreads();
  };
  for (int q = z0 - 2; q <= z1 + 1; q += 4) {
    step(integral_constant<int, 0>{}, q);
    step(integral_constant<int, 1>{}, q + 1);
    step(integral_constant<int, 2>{}, q + 2);
    step(integral_constant<int, 3>{}, q + 3);
  }
  cp_wait<0>();
  if (bad) atomicOr(a.flag, 1);
  if (!COARSE) block_sum<W::NT>(norm.total(), a.norm);
}

template <int TX>
constexpr size_t down_smem() {
  using W = Down<TX>;
  return sizeof(Ring<W::NT, 2 * W::PW>) + 7 * (size_t)W::PLANE * sizeof(long long);
}
template <int TX>
constexpr size_t up_smem() {
  using W = Up<TX>;
  return sizeof(Ring<W::NT, 1>) + 4 * (size_t)W::PLANE * sizeof(long long);
}

// F = a rho - b, rounded, less round(2 b_face 2^S) for each of the cell's fixed and
// open faces (c2 = 2^(S+1)), b = c *mu; per-block sums of F^2 without the
// faces' part (the norm of f).  Rounding to nearest gives regions of constant rho
// (the background of compact objects, less its mean) one and the same error, and
// an error that is smooth is what the inverse of L blows up: at 256^3, four
// blobs, it was most of the solution's.  So a rho - b is formed to 1/16 and rounded
// down after the addition of 0 .. 15 sixteenths, each to one cell of 16
// neighbouring ones, which makes their mean exact; red and black cells take
// halves of the offsets, so that what is left is as rough as it can be.
__global__ void __launch_bounds__(256) k_fx64_source(const double* rho,
                                                     long long* __restrict__ F, Grid g, Bc bc,
                                                     double a, double c, const double* mu, double c2,
                                                     double* __restrict__ partials) {
  dev::after_previous();
  const dev::Split sp(g.nx, g.ny);
  a *= 16.0;
  const double b = 16.0 * c * mu[0];
  const bool faces = bc.kind != BC_PERIODIC && bc.kind != BC_ZEROGRAD;
  SquareSum sum;
#pragma unroll 4
  for (long long t = blockIdx.x * 256LL + threadIdx.x; t < g.cells(); t += gridDim.x * 256LL) {
    // the last bits of i, i ^ j and i ^ j ^ k, and the next one of the latter
    const unsigned q = (unsigned)t, xy = q ^ q >> sp.lx, xyz = xy ^ q >> sp.lxy;
    const unsigned offset = (xyz & 1) << 3 | (xy & 1) << 2 | (q & 1) << 1 | (xyz >> 1 & 1);
    long long v = (cvt::d2ll_rn(fma(a, rho[t], -b)) + offset) >> 4;
    sum.add(v);
    if (faces) {
      int i, j, k;
      sp(t, i, j, k);
      if (i == 0 || i == g.nx - 1 || j == 0 || j == g.ny - 1 || k == 0 || k == g.nz - 1) {
        for (int s = 0; s < 6; ++s) {
          const int kind = face_kind(bc, s);
          if (kind != BC_FIXED && kind != BC_OPEN) continue;
          const int x = s < 2 ? i : s < 4 ? j : k, n = s < 2 ? g.nx : s < 4 ? g.ny : g.nz;
          if (x != ((s & 1) ? n - 1 : 0)) continue;
          v -= __double2ll_rn(
              dev::face_value(bc, g, s, (s < 2 ? j : i) + 1, (s < 4 ? k : j) + 1) * c2);
        }
      }
    }
    F[t] = v;
  }
  __shared__ double ws[8];
  double d = sum.total();
  for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = d;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) d += ws[w];
    partials[blockIdx.x] = d;
  }
}

// fc = 4 pi G (mean of rho over the eight children) - *mu: the source of the
// next level, straight from rho (one FP64 operation per cell).
__global__ void __launch_bounds__(256) k_fx64_restrict(const double* rho,
                                                       double* __restrict__ fc, Grid g, double c,
                                                       const double* mu) {
  dev::after_previous();
  const Grid gc{g.nx / 2, g.ny / 2, g.nz / 2};
  const dev::Split sp(gc.nx, gc.ny);
  const double m = mu[0];
  const size_t sy = g.nx, sz = (size_t)g.nx * g.ny;
  for (long long t = blockIdx.x * 256LL + threadIdx.x; t < gc.cells(); t += gridDim.x * 256LL) {
    int I, J, K;
    sp(t, I, J, K);
    const double* p = rho + dev::at(g, 2 * I, 2 * J, 2 * K);
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double* x = p + (q & 1) * sy + (q >> 1) * sz;
      v[q] = x[0] + x[1];
    }
    fc[t] = fma(0.125 * c, (v[0] + v[1]) + (v[2] + v[3]), -m);
  }
}

// phi = I' u (Sec. 2.3.1) on the integer grid, from the coarse level's doubles:
// weights 5, 30, -3 over 32 along x, y, z, rounded after each axis.  A thread
// marches up a chunk of cz coarse planes of one coarse column.
__global__ void __launch_bounds__(256) k_fx64_prolong(const double* uc, long long* __restrict__ out,
                                                      Grid g, Bc bc, int S, int cz,
                                                      long long items) {
  dev::after_previous();
  const Grid gc{g.nx / 2, g.ny / 2, g.nz / 2};
  const dev::Split sp(gc.nx, gc.ny);
  const size_t plane = (size_t)g.nx * g.ny;
  auto pair = [](long long a, long long b, long long c, long long& even, long long& odd) {
    const long long t = 30 * b + (a + c) + 16, d = 4 * (a - c);
    even = (t + d) >> 5;
    odd = (t - d) >> 5;
  };
  for (long long t = blockIdx.x * 256LL + threadIdx.x; t < items; t += gridDim.x * 256LL) {
    int I, J, ch;
    sp(t, I, J, ch);
    auto xy = [&](int K, long long o[2][2]) {
      long long v[3][2];
#pragma unroll
      for (int y = 0; y < 3; ++y) {
        long long e[3];
#pragma unroll
        for (int x = 0; x < 3; ++x)
          e[x] = cvt::d2ll_pow2_rn(dev::fetch(uc, I + x - 1, J + y - 1, K, gc, bc), S);
        pair(e[0], e[1], e[2], v[y][0], v[y][1]);
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) pair(v[0][x], v[1][x], v[2][x], o[0][x], o[1][x]);
    };
    const int K0 = ch * cz, K1 = min(K0 + cz, gc.nz);
    long long pm[2][2], p0[2][2], pp[2][2];
    xy(K0 - 1, pm);
    xy(K0, p0);
    for (int K = K0; K < K1; ++K) {
      xy(K + 1, pp);
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        long long lo[2], hi[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          pair(pm[y][x], p0[y][x], pp[y][x], lo[x], hi[x]);
          pm[y][x] = p0[y][x];
          p0[y][x] = pp[y][x];
        }
        const size_t q = dev::at(g, 2 * I, 2 * J + y, 2 * K);
        *reinterpret_cast<longlong2*>(out + q) = make_longlong2(lo[0], lo[1]);
        *reinterpret_cast<longlong2*>(out + q + plane) = make_longlong2(hi[0], hi[1]);
      }
    }
  }
}

// out[0] = sum of a[0 .. n) + sum of b[0 .. n), in a fixed order; out[1] = *flag.
__global__ void k_fx64_norm(const double* a, const double* b, int n, const int* flag, double* out) {
  dev::after_previous();
  __shared__ double ws[8];
  double s = 0.0;
#pragma unroll 4
  for (int t = threadIdx.x; t < n; t += 256) s += a[t] + b[t];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int w = 0; w < 8; ++w) r += ws[w];
    out[0] = r;
    out[1] = (double)*flag;
  }
}

Weight weight_of(double omega) {
  const double x = std::ldexp(omega / 6.0, 32), hi = std::nearbyint(x);  // x - hi is exact
  const double lo = std::nearbyint(std::ldexp(x - hi, 32));
  return Weight{(int)hi, lo >= 2147483647.0 ? 2147483647 : (int)lo};
}

template <typename K>
cudaError_t launch_leg(K* kernel, std::atomic<int>* configured, size_t smem, int threads, int tx,
                       const Fx64Args& a, cudaStream_t s) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev].load()) {
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev].store(1);
  }
  const dim3 grid(a.g.nx / tx, a.g.ny / TY, (a.g.nz + a.cz - 1) / a.cz);
  ++g_launches;
  const cudaError_t e = launch_after(kernel, grid, threads, smem, s, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <bool WALLS, int TX, bool COARSE>
cudaError_t launch(const Fx64Args& a, bool down, cudaStream_t s) {
  static std::atomic<int> configured[2][64];
  if (down)
    return launch_leg(k_fx64_down<WALLS, TX, COARSE>, configured[0], down_smem<TX>(), Down<TX>::NT,
                      TX, a, s);
  return launch_leg(k_fx64_up<WALLS, TX, COARSE>, configured[1], up_smem<TX>(), Up<TX>::NT, TX, a,
                    s);
}

// Tile width: 64 cells, or on levels that would leave SMs without a CTA, 32 cells
// (more halo, shorter chains); one CTA per SM either way, so that the threads of the
// narrow tiles (400, at most 128 CTAs of at least four planes) may have the
// registers they ask for: held to two CTAs they spilled 100-190 bytes, 64^3 fixed
// 1560 us instead of 1394.  Solves with the wide tiles at 64^3 as well, as here, and
// with the narrow ones up to 128^3 (GB300, periodic, us): 64^3 966, 889, 890; 128^3
// 1514, 1477, 1526; 256^3 4830, 4791, 4946.
int tile_width(Grid g) { return g.cells() <= (1LL << 18) ? 32 : 64; }

}  // namespace

bool fx64_ok(Grid g) {
  return g.nx % 64 == 0 && g.ny % TY == 0 && g.nz % 2 == 0 && g.nz >= 16 &&
         g.cells() <= (1LL << 30) && fx64_blocks(g) <= kPartials;
}

// Planes per CTA: the even count for which the last wave of CTAs is best filled,
// counting the six planes a chunk's halo costs; at most 128.
int fx64_cz(Grid g) {
  const int tx = tile_width(g), wave = sm_count();
  const long long cols = (long long)(g.nx / tx) * (g.ny / TY);
  int best = 0;
  long long least = 0;
  for (int cz = 4; cz <= 128 && cz <= g.nz; cz += 2) {
    const long long ctas = cols * ((g.nz + cz - 1) / cz);
    if (ctas > kPartials) continue;
    const long long cost = (ctas + wave - 1) / wave * (cz + 6);
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
  return (int)((long long)(g.nx / tile_width(g)) * (g.ny / TY) * ((g.nz + cz - 1) / cz));
}

static int face_kinds_of(const Bc& hom) {
  int fk = 0;
  for (int q = 0; q < 6; ++q) fk |= face_kind(hom, q) << (2 * q);
  return fk;
}

cudaError_t launch_fx64(const Fx64Leg& q, bool down, cudaStream_t s) {
  Fx64Args a{};
  a.u_in = q.u_in;
  a.u_out = q.u_out;
  a.F = q.F;
  a.g = q.g;
  a.fk = face_kinds_of(q.hom);
  a.cz = fx64_cz(q.g);
  a.w = weight_of(q.omega);
  a.norm = q.norm;
  a.fc = q.fc;
  a.fci = q.fci;
  a.ec = q.ec;
  // with |ec| < 2^56 and its sums of weight 64 below 2^62
  a.limit = q.coarse ? kFx64Correction : 59;
  a.flag = q.flag;
  const bool wide = tile_width(q.g) == 64;
  if (q.coarse) {
    if (a.fk) return wide ? launch<true, 64, true>(a, down, s) : launch<true, 32, true>(a, down, s);
    return wide ? launch<false, 64, true>(a, down, s) : launch<false, 32, true>(a, down, s);
  }
  if (a.fk) return wide ? launch<true, 64, false>(a, down, s) : launch<true, 32, false>(a, down, s);
  return wide ? launch<false, 64, false>(a, down, s) : launch<false, 32, false>(a, down, s);
}

cudaError_t launch_fx64_source(const double* rho, long long* F, Grid g, const Bc& bc,
                               double four_pi_G, const double* mu, double c, double two_pow_S,
                               double* partials, cudaStream_t s) {
  ++g_launches;
  launch_after(k_fx64_source, reduce_blocks(g.cells()), 256, 0, s, rho, F, g, bc, four_pi_G * c, c,
               mu, 2.0 * two_pow_S, partials);
  return cudaGetLastError();
}

cudaError_t launch_fx64_restrict(const double* rho, double* fc, Grid g, double four_pi_G,
                                 const double* mu, cudaStream_t s) {
  const long long b = (g.cells() / 8 + 255) / 256;
  ++g_launches;
  launch_after(k_fx64_restrict, (int)(b < 64LL * sm_count() ? b : 64LL * sm_count()), 256, 0, s, rho,
               fc, g, four_pi_G, mu);
  return cudaGetLastError();
}

cudaError_t launch_fx64_prolong(const double* uc, long long* phi, Grid g, const Bc& bc, int S,
                                cudaStream_t s) {
  // chunks of 8 coarse planes while that leaves four blocks per SM
  const long long cols = (long long)(g.nx / 2) * (g.ny / 2);
  const int nzc = g.nz / 2;
  int cz = 8;
  while (cz > 1 && cols * ((nzc + cz - 1) / cz) < 1024LL * sm_count()) cz /= 2;
  const long long items = cols * ((nzc + cz - 1) / cz), b = (items + 255) / 256;
  ++g_launches;
  launch_after(k_fx64_prolong, (int)(b < 64LL * sm_count() ? b : 64LL * sm_count()), 256, 0, s, uc,
               phi, g, bc, S, cz, items);
  return cudaGetLastError();
}

cudaError_t launch_fx64_norm(const double* red, const double* black, int nb, const int* flag,
                             double* out, cudaStream_t s) {
  ++g_launches;
  launch_after(k_fx64_norm, 1, 256, 0, s, red, black, nb, flag, out);
  return cudaGetLastError();
}

}  // namespace mg
