// mg_coarse.cu -- the coarse end of a V-cycle, or of the FMG ladder, in one
// launch.
//
// The levels of at most 16^3 cells are too small for a launch per half-sweep:
// what such a launch costs is its latency.  Here one launch runs whole
// V-cycles on all of them, with the levels in shared memory.
//
// FP32: one CTA of 1024 threads; the chain of passes is bound by latency, so
// each pass keeps its dependent chain short (the level's geometry ready in
// shared memory, sums as trees) and the levels of at most 64 cells, whose
// cycle from zero is a fixed linear map of their right-hand side, are one
// matrix-vector product with a matrix formed when the context is made.
//
// FP64: an SM issues two FP64 operations per clock, 64 clocks per warp
// instruction and scheduler, so one SM is too little for 16^3 cells.  A level
// of at least 16 planes along z is cut into 8 slabs, one per CTA of a cluster
// of 8, with one halo plane on either side; a CTA that updates a plane at the
// edge of its slab also stores it into its neighbour's halo plane through
// distributed shared memory, so that every load is local and a half-sweep
// ends with one cluster barrier (about 0.6 us).  The levels below (at most
// 8^3 on a cube) live in CTA 0, where a __syncthreads is enough.  The work is
// spread over full warps: a thread per fine cell prolongs (8 operations), two
// threads per coarse cell restrict (20 each).  FP32 levels of boxes that the
// fused legs do not take (a side below 32) are cut in the same way.
//
// A boundary value b on a face enters only at the top level, as the constant
// 2 b of the ghost 2 b - u: it is folded into the right-hand side while the
// level is loaded (f - 2 b / h^2), and every sweep then runs the homogeneous
// rule.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <atomic>
#include <utility>

#include "mg_device.cuh"
#include "mg_internal.h"

namespace cg = cooperative_groups;

namespace mg {
namespace {

template <typename T>
constexpr int kThreads = sizeof(T) == 4 ? 1024 : 512;

// One level as the kernel sees it; sizes are powers of two.  nx, ny, nz are
// the kernel's own axes (y and z exchanged when CoarseArgs::swap_yz).
template <typename T>
struct Level {
  int lx, ly, lz;  // log2 of the cells per axis
  int dist;        // cut into slabs over the cluster (else whole, in CTA 0)
  int u, f;        // offsets in shared memory (values of T); u of plane 0 of the slab
  T cf, ih2;       // -omega h^2 / 6, 1 / h^2
};

template <typename T>
struct CoarseArgs {
  Level<T> lev[kCoarseLevels];
  T* u_top;
  const T* f_top;
  long long sy, sz;  // strides of the top level's arrays along the kernel's y and z
  T cu, cs, cf0;     // 1 - omega, omega / 6; -h^2 / 6 of level 0 (its Gauss-Seidel sweeps)
  int top, pre, post, cycles;
  int zero_guess;    // the first cycle starts from u = 0 (else from u_top)
  int fk_top, fk;    // kind of each face (2 bits), kernel's axes: top level, levels below
  int swap_yz;
  const T* dense;    // kDense x kDense matrix of the cycle on level dense_level (0: none)
  int dense_level;
  int nmax0;         // sweeps on a level 0 of several cells
  double h[kCoarseLevels];
  Bc bc[kCoarseLevels];  // physical rules (FMG: every level; else the top's only)
};

__device__ __forceinline__ int fkind(int fk, int q) { return (fk >> (2 * q)) & 3; }

// A level's cells of this CTA: planes [k0, k0 + P).  off[q] and neg[q]: where
// a neighbour across that end of the slab is (a halo plane, the periodic
// image, or for a wall the cell itself), and whether it enters with a minus
// sign (zero fixed).
template <typename T>
struct Slab {
  int lx, ly, P, k0, sy, sz;
  int u, f;  // offsets in shared memory
  int off[6];
  int neg;   // bit q
  int dist;
  T cf, ih2;
};

template <typename T, bool PER>
struct Prog {
  static constexpr int kT = kThreads<T>;
  const CoarseArgs<T>& a;
  T* sm;
  Slab<T> (*slabs)[kCoarseLevels];  // [1]: the level as the top of a cycle
  cg::cluster_group cl;
  int rank, nct;
  T m[kDense * kDense / kT];  // this thread's entries of the dense levels' matrix

  __device__ Prog(const CoarseArgs<T>& a_, T* sm_, Slab<T> (*slabs_)[kCoarseLevels])
      : a(a_), sm(sm_), slabs(slabs_), cl(cg::this_cluster()), rank((int)cl.block_rank()),
        nct((int)cl.num_blocks()) {
    const int t = threadIdx.x;
    if (t < 2 * (a.top + 1)) make_slab(t >> 1, t & 1 ? a.fk_top : a.fk, slabs[t & 1][t >> 1]);
    if (a.dense_level > 0 && rank == 0) {
      // entry (row, col): row t / kSeg, columns from (t % kSeg) kDense / kSeg
#pragma unroll
      for (int q = 0; q < kDense * kDense / kT; ++q) m[q] = a.dense[t * (kDense * kDense / kT) + q];
    }
  }

  __device__ void make_slab(int l, int fk, Slab<T>& s) const {
    const Level<T>& v = a.lev[l];
    const int nz = 1 << v.lz;
    s.lx = v.lx;
    s.ly = v.ly;
    s.dist = v.dist;
    s.P = v.dist ? nz / nct : nz;
    s.k0 = v.dist ? rank * s.P : 0;
    s.sy = 1 << v.lx;
    s.sz = 1 << (v.lx + v.ly);
    s.u = v.u;
    s.f = v.f;
    s.cf = v.cf;
    s.ih2 = v.ih2;
    s.neg = 0;
    const int w[3] = {(1 << v.lx) - 1, ((1 << v.ly) - 1) * s.sy, (s.P - 1) * s.sz};
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int ax = q >> 1, kind = fkind(fk, q);
      const bool hi = q & 1;
      if (ax == 2 && s.dist && (kind == BC_PERIODIC || (hi ? s.k0 + s.P < nz : s.k0 > 0))) {
        s.off[q] = hi ? s.sz : -s.sz;  // the halo plane
        continue;
      }
      s.off[q] = kind != BC_PERIODIC ? 0 : hi ? -w[ax] : w[ax];
      if (kind == BC_FIXED) s.neg |= 1 << q;
    }
  }

  __device__ __forceinline__ void sync(const Slab<T>& s) const {
    if (s.dist) cl.sync();
    else __syncthreads();
  }
  __device__ __forceinline__ void sync_all() const {
    if (nct > 1) cl.sync();
    else __syncthreads();
  }
  // The CTAs that run a level's steps.
  __device__ __forceinline__ bool mine(int l) const { return a.lev[l].dist || rank == 0; }

  // Store v at cell c (plane p) and into the neighbours' halo planes.  The
  // neighbour across a wall gets a value that it never reads.
  __device__ __forceinline__ void put(const Slab<T>& s, int c, int p, T v) const {
    T* u = sm + s.u;
    u[c] = v;
    if (!s.dist) return;
    if (p == 0) {
      T* r = cl.map_shared_rank(u, rank == 0 ? nct - 1 : rank - 1);
      r[c + s.P * s.sz] = v;
    }
    if (p == s.P - 1) {
      T* r = cl.map_shared_rank(u, rank == nct - 1 ? 0 : rank + 1);
      r[c - s.P * s.sz] = v;
    }
  }

  // The neighbour of cell c at distance `step`, or across an end (its offset
  // and sign).
  __device__ __forceinline__ T nb(const T* u, int c, bool inside, int step, int off,
                                  int neg) const {
    T v = u[c + (inside ? step : off)];
    if (!PER)
      if (!inside && neg) v = -v;
    return v;
  }
  __device__ __forceinline__ T nb(const Slab<T>& s, const T* u, int c, bool inside, int step,
                                  int q) const {
    return nb(u, c, inside, step, s.off[q], s.neg >> q & 1);
  }

  // One colour of SMOOTH (Eqs. rbsor1-rbsor2).
  __device__ __forceinline__ void half_sweep(const Slab<T>& s, int colour, T cu, T cs, T cf) const {
    const T *u = sm + s.u, *f = sm + s.f;
    const int half = (s.P << (s.lx + s.ly)) >> 1, wx = (1 << s.lx) - 1, wy = (1 << s.ly) - 1;
    for (int t = threadIdx.x; t < half; t += kT) {
      const int r = t >> (s.lx - 1), j = r & wy, p = r >> s.ly;
      const int i = 2 * (t & (wx >> 1)) + ((j + s.k0 + p + colour) & 1);
      const int c = (r << s.lx) + i;
      const T sx = nb(s, u, c, i > 0, -1, 0) + nb(s, u, c, i < wx, 1, 1);
      const T sy = nb(s, u, c, j > 0, -s.sy, 2) + nb(s, u, c, j < wy, s.sy, 3);
      const T sz = nb(s, u, c, p > 0, -s.sz, 4) + nb(s, u, c, p < s.P - 1, s.sz, 5);
      put(s, c, p, cs * ((sx + sy) + sz) + (cu * u[c] + cf * f[c]));
    }
    sync(s);
  }

  // A cell's value after the red half-sweep from u = 0 (red cells cf f, black
  // cells 0), or 0 where no sweep follows.
  __device__ __forceinline__ T zero_red(int i, int j, int k, T cf, T fv, bool sweep) const {
    return sweep && !((i + j + k) & 1) ? cf * fv : T(0);
  }

  // `steps` SMOOTH steps; red0: the first red half-sweep is done already.
  __device__ __forceinline__ void smooth(const Slab<T>& s, int steps, bool red0) const {
    for (int q = red0 ? 1 : 0; q < 2 * steps; ++q) half_sweep(s, q & 1, a.cu, a.cs, s.cf);
  }

  // f of level l - 1 = mean over the eight children of f - L u (Algorithm 1,
  // steps 2-3), and that level's start u = 0 with its first red half-sweep.
  // The sum over the children of the neighbour sums is three times the sum of
  // the eight cells (each has three neighbours among them) plus the 24 cells
  // around the block.  kHalf: two neighbouring lanes share a block, a plane
  // each (FP64, bound by its units); otherwise a thread has the whole block
  // (FP32, bound by instructions and shared-memory wavefronts).
  static constexpr bool kHalf = sizeof(T) == 8;

  __device__ __forceinline__ void defect_restrict(const Slab<T>& s, int l) const {
    const Slab<T> sc = slabs[0][l - 1];
    const int lxy = sc.lx + sc.ly, kc0 = s.k0 >> 1;
    const bool remote = s.dist && !sc.dist;  // the coarse level lives in CTA 0
    const int at0 = sc.dist ? 0 : kc0;       // coarse plane index of the first one here
    T* to = remote ? cl.map_shared_rank(sm, 0) : sm;
    const bool sweep = a.pre > 0 && l - 1 > 0;
    const int wx = (1 << s.lx) - 1, wy = (1 << s.ly) - 1;
    const T *u = sm + s.u, *f = sm + s.f;
    const int work = (s.P << lxy) >> (kHalf ? 0 : 1);
    for (int t = threadIdx.x; t < ((work + 31) & ~31); t += kT) {
      const bool live = t < work;
      const int b = live ? (kHalf ? t >> 1 : t) : 0;
      const int I = b & ((1 << sc.lx) - 1), J = (b >> sc.lx) & ((1 << sc.ly) - 1), K = b >> lxy;
      // f - L u summed over the block's cells in plane 2 K + d
      auto plane = [&](int d) {
        const int i = 2 * I, j = 2 * J, p = 2 * K + d;
        const int c = (p << (s.lx + s.ly)) + (j << s.lx) + i, cy = c + s.sy;
        const T own = (u[c] + u[c + 1]) + (u[cy] + u[cy + 1]);
        const T fs = (f[c] + f[c + 1]) + (f[cy] + f[cy + 1]);
        const T ox = (nb(s, u, c, i > 0, -1, 0) + nb(s, u, cy, i > 0, -1, 0)) +
                     (nb(s, u, c + 1, i + 1 < wx, 1, 1) + nb(s, u, cy + 1, i + 1 < wx, 1, 1));
        const T oy =
            (nb(s, u, c, j > 0, -s.sy, 2) + nb(s, u, c + 1, j > 0, -s.sy, 2)) +
            (nb(s, u, cy, j + 1 < wy, s.sy, 3) + nb(s, u, cy + 1, j + 1 < wy, s.sy, 3));
        const bool in = d ? p < s.P - 1 : p > 0;
        const int st = d ? s.sz : -s.sz, off = d ? s.off[5] : s.off[4];
        const int neg = s.neg >> (4 + d) & 1;
        const T oz = (nb(u, c, in, st, off, neg) + nb(u, c + 1, in, st, off, neg)) +
                     (nb(u, cy, in, st, off, neg) + nb(u, cy + 1, in, st, off, neg));
        return fs - s.ih2 * (((ox + oy) + oz) - T(3) * own);
      };
      T fv;
      if (kHalf) {
        fv = plane(t & 1);
        fv += __shfl_xor_sync(0xffffffffu, fv, 1);
        if (t & 1) continue;
      } else {
        fv = plane(0) + plane(1);
      }
      if (!live) continue;
      fv *= T(0.125);
      const int cc = ((at0 + K) << lxy) + (J << sc.lx) + I;
      to[sc.f + cc] = fv;
      const T uv = zero_red(I, J, kc0 + K, sc.cf, fv, sweep);
      if (sc.dist) put(sc, cc, K, uv);
      else to[sc.u + cc] = uv;
    }
    sync(s);
  }

  // u_l += trilinear(u_{l-1}) (Algorithm 1, steps 5-6).
  __device__ __forceinline__ void prolong(const Slab<T>& s, int l) const {
    if (sizeof(T) == 8) prolong_cells(s, slabs[0][l - 1]);
    else prolong_blocks(s, slabs[0][l - 1]);
    sync(s);
  }

  // A thread per coarse cell (FP32: fewest instructions per fine cell): the
  // coarse values around it interpolated along x, then y, then z.
  __device__ __forceinline__ void prolong_blocks(const Slab<T>& s, const Slab<T>& c) const {
    const int n = s.P >> 1, kc0 = c.dist ? 0 : s.k0 >> 1;
    const int wx = (1 << c.lx) - 1, wy = (1 << c.ly) - 1;
    const T* uc = sm + c.u;
    T* u = sm + s.u;
    for (int t = threadIdx.x; t < n << (c.lx + c.ly); t += kT) {
      const int I = t & wx, J = (t >> c.lx) & wy, q = t >> (c.lx + c.ly), K = kc0 + q;
      const int o = (K << (c.lx + c.ly)) + (J << c.lx) + I;
      int ox[3], oy[3], oz[3];
      bool nx[3], ny[3], nz[3];
      ox[1] = oy[1] = oz[1] = 0;
      nx[1] = ny[1] = nz[1] = false;
      ox[0] = I > 0 ? -1 : c.off[0];
      ox[2] = I < wx ? 1 : c.off[1];
      oy[0] = J > 0 ? -c.sy : c.off[2];
      oy[2] = J < wy ? c.sy : c.off[3];
      oz[0] = K > 0 ? -c.sz : c.off[4];
      oz[2] = K < c.P - 1 ? c.sz : c.off[5];
      nx[0] = I == 0 && (c.neg & 1);
      nx[2] = I == wx && (c.neg & 2);
      ny[0] = J == 0 && (c.neg & 4);
      ny[2] = J == wy && (c.neg & 8);
      nz[0] = K == 0 && (c.neg & 16);
      nz[2] = K == c.P - 1 && (c.neg & 32);
      T vy[3][2][2];
#pragma unroll
      for (int z = 0; z < 3; ++z) {
        T vx[3][2];
#pragma unroll
        for (int y = 0; y < 3; ++y) {
          T v[3];
#pragma unroll
          for (int x = 0; x < 3; ++x) {
            v[x] = uc[o + ox[x] + oy[y] + oz[z]];
            if (!PER && (nx[x] != ny[y]) != nz[z]) v[x] = -v[x];
          }
          dev::interp1<T, false>(v[0], v[1], v[2], vx[y][0], vx[y][1]);
        }
#pragma unroll
        for (int x = 0; x < 2; ++x)
          dev::interp1<T, false>(vx[0][x], vx[1][x], vx[2][x], vy[z][0][x], vy[z][1][x]);
      }
#pragma unroll
      for (int y = 0; y < 2; ++y)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          T lo, hi;
          dev::interp1<T, false>(vy[0][y][x], vy[1][y][x], vy[2][y][x], lo, hi);
          const int w = (2 * q << (s.lx + s.ly)) + ((2 * J + y) << s.lx) + 2 * I + x;
          put(s, w, 2 * q, u[w] + lo);
          put(s, w + s.sz, 2 * q + 1, u[w + s.sz] + hi);
        }
    }
  }

  // A thread per fine cell (FP64: full warps on its units): 27/64 of its
  // parent, 9/64 of the three nearest along an axis, 3/64 and 1/64 of those
  // across an edge and the corner.
  __device__ __forceinline__ void prolong_cells(const Slab<T>& s, const Slab<T>& c) const {
    const T *uc = sm + c.u, *u = sm + s.u;
    const int kc0 = c.dist ? 0 : s.k0 >> 1;
    const int wx = (1 << s.lx) - 1, wy = (1 << s.ly) - 1;
    for (int t = threadIdx.x; t < s.P << (s.lx + s.ly); t += kT) {
      const int i = t & wx, r = t >> s.lx, j = r & wy, p = r >> s.ly;
      const int I = i >> 1, J = j >> 1, K = kc0 + (p >> 1);
      const int o = (K << (c.lx + c.ly)) + (J << c.lx) + I;
      const bool ex = (i & 1) ? i == wx : i == 0, ey = (j & 1) ? j == wy : j == 0,
                 ez = (p & 1) ? K == c.P - 1 : K == 0;
      const int qx = i & 1, qy = 2 + (j & 1), qz = 4 + (p & 1);
      const int dx = ex ? ((i & 1) ? c.off[1] : c.off[0]) : 2 * (i & 1) - 1;
      const int dy = ey ? ((j & 1) ? c.off[3] : c.off[2]) : (j & 1) ? c.sy : -c.sy;
      const int dz = ez ? ((p & 1) ? c.off[5] : c.off[4]) : (p & 1) ? c.sz : -c.sz;
      const bool nx = !PER && ex && (c.neg >> qx & 1), ny = !PER && ey && (c.neg >> qy & 1),
                 nz = !PER && ez && (c.neg >> qz & 1);
      const T c0 = uc[o];
      T cx = uc[o + dx], cy = uc[o + dy], cz = uc[o + dz];
      T cxy = uc[o + dx + dy], cxz = uc[o + dx + dz], cyz = uc[o + dy + dz];
      T cxyz = uc[o + dx + dy + dz];
      if (!PER) {
        cx = nx ? -cx : cx;
        cy = ny ? -cy : cy;
        cz = nz ? -cz : cz;
        cxy = nx != ny ? -cxy : cxy;
        cxz = nx != nz ? -cxz : cxz;
        cyz = ny != nz ? -cyz : cyz;
        cxyz = (nx != ny) != nz ? -cxyz : cxyz;
      }
      const T v = T(27.0 / 64) * c0 + T(9.0 / 64) * ((cx + cy) + cz);
      const T w = T(3.0 / 64) * ((cxy + cxz) + cyz) + (T(1.0 / 64) * cxyz + u[t]);
      put(s, t, p, v + w);
    }
  }

  // COARSEST in CTA 0: one cell exactly, several by Gauss-Seidel sweeps from 0.
  __device__ __forceinline__ void coarsest(int fk) const {
    const Slab<T> s = slabs[fk == a.fk ? 0 : 1][0];
    if (s.lx == 0) {
      if (threadIdx.x == 0) {
        int walls = 0;
        for (int q = 0; q < 6; ++q) walls += !PER && fkind(fk, q) == BC_FIXED;
        sm[s.u] = walls ? (T)(-a.h[0] * a.h[0] * (double)sm[s.f] / (2.0 * walls)) : T(0);
      }
      __syncthreads();
      return;
    }
    // u is 0 here: set with the restricted f, or below in the FMG ladder
    for (int q = 0; q < 2 * a.nmax0; ++q) half_sweep(s, q & 1, T(0), T(1.0 / 6.0), a.cf0);
  }

  // u = M f on the dense level: kSeg lanes per row.
  __device__ __forceinline__ void dense_cycle() const {
    constexpr int kPer = kDense * kDense / kT, kSeg = kDense / kPer;
    const Slab<T> s = slabs[0][a.dense_level];
    const int row = threadIdx.x / kSeg, col = (threadIdx.x % kSeg) * kPer;
    const T* f = sm + s.f + col;
    T v = m[0] * f[0];
#pragma unroll
    for (int q = 1; q < kPer; ++q) v += m[q] * f[q];
#pragma unroll
    for (int o = kSeg / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x % kSeg == 0) sm[s.u + row] = v;
    __syncthreads();
  }

  // One V-cycle on levels top .. 0 (Algorithm 1).  red0: the top's first red
  // half-sweep is done (a start from 0).
  __device__ __forceinline__ void vcycle(int top, bool red0) const {
    const int dl = a.dense_level < top ? a.dense_level : 0;
    for (int l = top; l > dl; --l) {
      if (!mine(l)) continue;
      const Slab<T> s = slabs[l == top][l];
      smooth(s, a.pre, l < top || red0);
      defect_restrict(s, l);
    }
    if (rank == 0) {
      if (dl > 0) dense_cycle();
      else coarsest(a.fk);
    }
    for (int l = dl + 1; l <= top; ++l) {
      if (a.lev[l].dist && !a.lev[l - 1].dist) {
        // hand the level below, complete in CTA 0, to every CTA
        if (rank == 0) {
          const Level<T>& v = a.lev[l - 1];
          const int n = 1 << (v.lx + v.ly + v.lz);
          for (int t = threadIdx.x; t < n; t += kT) {
            const T x = sm[v.u + t];
            for (int r = 1; r < nct; ++r) cl.map_shared_rank(sm, r)[v.u + t] = x;
          }
        }
        cl.sync();
      }
      if (!mine(l)) continue;
      const Slab<T> s = slabs[l == top][l];
      prolong(s, l);
      smooth(s, a.post, false);
    }
  }

  // Global index of cell (i, j, k) of the top level (kernel's axes).
  __device__ __forceinline__ long long gat(int i, int j, int k) const {
    return i + j * a.sy + k * a.sz;
  }

  // What the boundary values of cell (i, j, k)'s faces add to its six
  // neighbours' sum under the physical rule bc of a level of size g: 2 b per
  // fixed or open face.  Axes as in the level's own array.
  __device__ static double face_terms(const Bc& bc, const Grid& g, int i, int j, int k) {
    if (bc.kind == BC_PERIODIC || bc.kind == BC_ZEROGRAD) return 0.0;
    double b = 0.0;
    for (int q = 0; q < 6; ++q) {
      const int kind = face_kind(bc, q);
      if (kind != BC_FIXED && kind != BC_OPEN) continue;
      const int x = q < 2 ? i : q < 4 ? j : k, n = q < 2 ? g.nx : q < 4 ? g.ny : g.nz;
      if (x != ((q & 1) ? n - 1 : 0)) continue;
      b += 2.0 * dev::face_value(bc, g, q, (q < 2 ? j : i) + 1, (q < 4 ? k : j) + 1);
    }
    return b;
  }

  __device__ void run_vcycles() const {
    const int top = a.top;
    const Slab<T> s = slabs[1][top];
    const int cells = s.P << (s.lx + s.ly), nz = 1 << a.lev[top].lz;
    T *u = sm + s.u, *f = sm + s.f;
    const bool red0 = a.zero_guess != 0;
    if (mine(top)) {
      const Bc& bc = a.bc[top];
      const bool fold = bc.kind == BC_OPEN || (bc.kind == BC_FIXED && bc.value != 0.0) ||
                        (bc.kind == BC_MIXED && bc.faces);
      const Grid g{s.sy, a.swap_yz ? nz : 1 << s.ly, a.swap_yz ? 1 << s.ly : nz};
#pragma unroll 4
      for (int t = threadIdx.x; t < cells; t += kT) {
        const int i = t & (s.sy - 1), r = t >> s.lx, j = r & ((1 << s.ly) - 1), p = r >> s.ly;
        T x = a.f_top[gat(i, j, s.k0 + p)];
        if (fold) {
          const double b = a.swap_yz ? face_terms(bc, g, i, s.k0 + p, j)
                                     : face_terms(bc, g, i, j, s.k0 + p);
          if (b != 0.0) x = (T)((double)x - b / (a.h[top] * a.h[top]));
        }
        f[t] = x;
        if (red0) put(s, t, p, zero_red(i, j, s.k0 + p, s.cf, x, a.pre > 0));
      }
      if (!red0) {  // u with its halo planes (a wall's is never read)
        const int lo = s.dist ? -1 : 0, planes = s.dist ? s.P + 2 : s.P;
#pragma unroll 4
        for (int t = threadIdx.x; t < planes << (s.lx + s.ly); t += kT) {
          const int i = t & (s.sy - 1), r = t >> s.lx, j = r & ((1 << s.ly) - 1);
          const int p = (r >> s.ly) + lo, k = (s.k0 + p) & (nz - 1);
          u[p * s.sz + (t & (s.sz - 1))] = a.u_top[gat(i, j, k)];
        }
      }
    }
    sync_all();
    for (int q = 0; q < a.cycles; ++q) vcycle(top, q == 0 && red0);
    if (mine(top))
      for (int t = threadIdx.x; t < cells; t += kT) {
        const int i = t & (s.sy - 1), r = t >> s.lx, j = r & ((1 << s.ly) - 1), p = r >> s.ly;
        a.u_top[gat(i, j, s.k0 + p)] = u[t];
      }
    // no CTA leaves while another could still store into its shared memory
    sync_all();
  }

  // Algorithm 2 on levels 0 .. top in one CTA (no level is cut into slabs).
  __device__ void run_fmg() const {
    for (int l = a.top; l >= 0; --l) {
      const Level<T>& v = a.lev[l];
      const Grid g{1 << v.lx, 1 << v.ly, 1 << v.lz};
      if (l == a.top)
        for (int t = threadIdx.x; t < (int)g.cells(); t += kT) sm[v.f + t] = a.f_top[t];
      __syncthreads();
      if (l > 0) dev::restrict_range(sm + v.f, sm + a.lev[l - 1].f, g, threadIdx.x, kT);
      __syncthreads();
      for (int t = threadIdx.x; t < (int)g.cells(); t += kT) {
        const int i = t & (g.nx - 1), j = (t >> v.lx) & (g.ny - 1), k = t >> (v.lx + v.ly);
        const double b = face_terms(a.bc[l], g, i, j, k);
        if (b != 0.0) sm[v.f + t] = (T)((double)sm[v.f + t] - b / (a.h[l] * a.h[l]));
        if (l == 0) sm[v.u + t] = T(0);
      }
      __syncthreads();
    }
    coarsest(a.fk_top);
    for (int l = 1; l <= a.top; ++l) {
      const Level<T>& v = a.lev[l];
      const Grid g{1 << v.lx, 1 << v.ly, 1 << v.lz};
      dev::prolong_range<T, true>(sm + a.lev[l - 1].u, sm + v.u, g, a.bc[l - 1], 0, threadIdx.x,
                                  kT);
      __syncthreads();
      vcycle(l, false);
    }
    const Level<T>& v = a.lev[a.top];
    for (int t = threadIdx.x; t < 1 << (v.lx + v.ly + v.lz); t += kT) a.u_top[t] = sm[v.u + t];
  }

  // Column blockIdx.x of the dense level's matrix: a V-cycle from zero with
  // that unit vector as the right-hand side.
  __device__ void run_basis() const {
    const Slab<T> s = slabs[1][a.top];
    const int n = s.P << (s.lx + s.ly), b = blockIdx.x;
    for (int t = threadIdx.x; t < n; t += kT) {
      const int i = t & (s.sy - 1), r = t >> s.lx, j = r & ((1 << s.ly) - 1), k = r >> s.ly;
      const T x = t == b ? T(1) : T(0);
      sm[s.f + t] = x;
      sm[s.u + t] = zero_red(i, j, k, s.cf, x, a.pre > 0);
    }
    __syncthreads();
    vcycle(a.top, true);
    for (int t = threadIdx.x; t < n; t += kT) a.u_top[t * kDense + b] = sm[s.u + t];
  }
};

template <typename T, bool PER, int MODE>
__global__ void __launch_bounds__(kThreads<T>) k_coarse(const __grid_constant__ CoarseArgs<T> a) {
  // a CTA's shared memory may be stored into once that CTA has started: the
  // cluster meets before the first put().  Arriving first, waiting last, the
  // barrier passes while the kernel before this one runs and the slabs are made.
  cg::cluster_group cl = cg::this_cluster();
  auto started = cl.barrier_arrive();
  dev::after_previous();
  extern __shared__ double coarse_smem[];
  __shared__ Slab<T> slabs[2][kCoarseLevels];
  Prog<T, PER> p(a, reinterpret_cast<T*>(coarse_smem), slabs);
  __syncthreads();
  cl.barrier_wait(std::move(started));
  if constexpr (MODE == COARSE_FMG) p.run_fmg();
  else if constexpr (MODE == COARSE_BASIS) p.run_basis();
  else p.run_vcycles();
}

// ---------------------------------------------------------------------------
// The same cycles in FP32 for a cube of 16^3 cells, the coarse end of every
// cubic grid of the mixed path.  Here the sizes are compile-time constants and
// a thread owns half a row of the 16^3 level (and the first 64 a row of 8^3)
// for the whole call: its u and f stay in registers, the colours of a row are
// kept apart (four red, four black per half row), and shared memory carries
// only what the neighbouring rows read, in 16-byte loads: four per half-step
// of four cells, and one shuffle for the cell across the half row's end.  A
// half-step is about 45 instructions per thread where the general program
// above spends about 240 on the same four cells (14-19 us per launch).
//
// Cell i = 2 m + e of row (j, k), e = (j + k) & 1, is red cell m of the row;
// 2 m + 1 - e is black cell m.  A row's planes are padded so that the eight
// lanes of a 16-byte phase (half row, j & 1, k & 1) hit different banks.

struct CubeArgs {
  float* u;
  const float* f;
  const float* dense;
  float cu, cs;
  float cf[2], ih2[2];  // levels 8^3, 16^3
  int fk_top, fk;
  int pre, post, cycles, zero_guess;
};

constexpr int kCubeThreads = 512;

// Where a thread's row has its neighbour rows y-, y+, z-, z+: offset of that
// row, or for a wall of the row itself with the ghost's sign.
struct Rows {
  int o[4];
  float s[4];
  bool wall[4];
};

template <int N, bool PER>
__device__ __forceinline__ Rows rows_of(int fk, int j, int k, int sj, int sk, int tail) {
  Rows r;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const bool hi = q & 1;
    const int x = q < 2 ? j : k, kind = PER ? (int)BC_PERIODIC : fkind(fk, 2 + q);
    const bool end = x == (hi ? N - 1 : 0);
    r.wall[q] = !PER && end && kind != BC_PERIODIC;
    r.s[q] = r.wall[q] && kind == BC_FIXED ? -1.f : 1.f;
    const int y = r.wall[q] ? x : end ? (hi ? 0 : N - 1) : (hi ? x + 1 : x - 1);
    r.o[q] = (q < 2 ? y * sj + k * sk : j * sj + y * sk) + tail;
  }
  return r;
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// One colour of SMOOTH on four cells: own and oth the row's cells of that and
// of the other colour, x[m] the neighbour along x outside the pair, so / ss
// the shared arrays of the other and of the same colour.
template <bool PER>
__device__ __forceinline__ void relax4(float (&own)[4], const float (&oth)[4], const float (&x)[4],
                                       const float (&f)[4], const float* so, const float* ss,
                                       const Rows& r, float cu, float cs, float cf) {
  float4 v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = ld4((PER || !r.wall[q] ? so : ss) + r.o[q]);
  float s[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) s[m] = oth[m] + x[m];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
    for (int m = 0; m < 4; ++m) s[m] = PER ? s[m] + w[m] : fmaf(r.s[q], w[m], s[m]);
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) own[m] = cs * s[m] + (cu * own[m] + cf * f[m]);
}

// Defects summed over the pairs (2 m, 2 m + 1) of a row: xl, xr the cells
// outside each pair along x.
template <bool PER>
__device__ __forceinline__ void pair_defects(float (&d)[4], const float (&red)[4],
                                             const float (&blk)[4], const float (&xl)[4],
                                             const float (&xr)[4], const float (&fr)[4],
                                             const float (&fb)[4], const float* sr, const float* sb,
                                             const Rows& r, float ih2) {
  float s[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) s[m] = (xl[m] + xr[m]) - 5.f * (red[m] + blk[m]);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float4 a = ld4(sr + r.o[q]), b = ld4(sb + r.o[q]);
    const float w[4] = {a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w};
#pragma unroll
    for (int m = 0; m < 4; ++m) s[m] = PER ? s[m] + w[m] : fmaf(r.s[q], w[m], s[m]);
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) d[m] = (fr[m] + fb[m]) - ih2 * s[m];
}

// The coarse rows a fine row (j, k) is interpolated from, with their weights
// (times 16): its parent's, the nearer one along y, along z, and across.
struct Parents {
  int o[4];
  float w[4];
};
template <int NC, bool PER>
__device__ __forceinline__ Parents parents_of(int fk, int j, int k, int sj, int sk) {
  const int J = j >> 1, K = k >> 1;
  auto near = [&](int x, int hi, int q, float& s) {
    const int y = hi ? x + 1 : x - 1, kind = PER ? (int)BC_PERIODIC : fkind(fk, q + hi);
    s = 1.f;
    if (y >= 0 && y < NC) return y;
    if (kind == BC_PERIODIC) return hi ? 0 : NC - 1;
    if (kind == BC_FIXED) s = -1.f;
    return x;
  };
  float sy, sz;
  const int J2 = near(J, j & 1, 2, sy), K2 = near(K, k & 1, 4, sz);
  Parents p;
  p.o[0] = J * sj + K * sk;
  p.o[1] = J2 * sj + K * sk;
  p.o[2] = J * sj + K2 * sk;
  p.o[3] = J2 * sj + K2 * sk;
  p.w[0] = 9.f;
  p.w[1] = 3.f * sy;
  p.w[2] = 3.f * sz;
  p.w[3] = sy * sz;
  return p;
}

template <bool PER>
__global__ void __launch_bounds__(kCubeThreads) k_cube16(const __grid_constant__ CubeArgs a) {
  dev::after_previous();
  constexpr int S16 = 144, S8 = 48;  // padded plane strides (floats)
  __shared__ alignas(16) float sR[16 * S16], sB[16 * S16];
  __shared__ alignas(16) float cR[8 * S8], cB[8 * S8], cfR[8 * S8], cfB[8 * S8];
  __shared__ alignas(16) float nat[512], f4[kDense], u4[kDense];
  const int t = threadIdx.x;
  const int h = t & 1, j0 = t >> 1 & 1, k0 = t >> 2 & 1, J = t >> 3 & 7, K = t >> 6;
  const int j = 2 * J + j0, k = 2 * K + k0;
  const bool e = j0 != k0;
  const int own = k * S16 + j * 8 + 4 * h;
  const Rows rw = rows_of<16, PER>(a.fk_top, j, k, 8, S16, 4 * h);
  // x walls of this half row (sign of the ghost, 0: none)
  auto xsign = [&](int fk, int q) {
    const int kind = PER ? (int)BC_PERIODIC : fkind(fk, q);
    return kind == BC_PERIODIC ? 0.f : kind == BC_FIXED ? -1.f : 1.f;
  };
  const float wl = h == 0 ? xsign(a.fk_top, 0) : 0.f, wh = h == 1 ? xsign(a.fk_top, 1) : 0.f;
  float md[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) md[q] = a.dense[8 * t + q];
  float r[4], b[4], fr[4], fb[4];
  // natural order to colours: cells 8 h .. 8 h + 7 of the row
  const size_t g = ((size_t)k * 16 + j) * 16 + 8 * h;
  auto split = [&](const float* p, float (&red)[4], float (&blk)[4]) {
    const float4 lo = ld4(p), hi = ld4(p + 4);
    const float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      red[m] = e ? v[2 * m + 1] : v[2 * m];
      blk[m] = e ? v[2 * m] : v[2 * m + 1];
    }
  };
  split(a.f + g, fr, fb);
  if (a.zero_guess) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      r[m] = a.pre > 0 ? a.cf[1] * fr[m] : 0.f;
      b[m] = 0.f;
    }
  } else {
    split(a.u + g, r, b);
  }
  st4(sR + own, r);
  st4(sB + own, b);
  __syncthreads();
  // the cell across the end of the half row that colour `own` reads: up: the
  // other colour's m + 1 (from m = 3), else its m - 1 (from m = 0)
  auto sweep16 = [&](float (&o)[4], const float (&n)[4], const float (&f)[4], float* so, float* sn,
                     bool up) {
    float got = __shfl_xor_sync(0xffffffffu, up ? n[0] : n[3], 1);
    if (!PER) {
      if (up && wh != 0.f) got = wh * o[3];
      if (!up && wl != 0.f) got = wl * o[0];
    }
    float x[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) x[m] = up ? (m < 3 ? n[m + 1 & 3] : got) : (m > 0 ? n[m - 1 & 3] : got);
    relax4<PER>(o, n, x, f, sn, so, rw, a.cu, a.cs, a.cf[1]);
    st4(so + own, o);
    __syncthreads();
  };
  auto smooth16 = [&](int steps, bool red0) {
    for (int q = 0; q < steps; ++q) {
      if (q > 0 || !red0) sweep16(r, b, fr, sR, sB, e);
      sweep16(b, r, fb, sB, sR, !e);
    }
  };
  // the 8^3 level: the first 64 threads have a row each
  const int i8j = t & 1, i8k = t >> 1 & 1, J8 = t >> 2 & 3, K8 = t >> 4 & 3;
  const int j8 = 2 * J8 + i8j, k8 = 2 * K8 + i8k;
  const bool e8 = i8j != i8k;
  const int own8 = k8 * S8 + j8 * 4;
  const Rows rw8 = rows_of<8, PER>(a.fk, j8, k8, 4, S8, 0);
  const float xl8 = xsign(a.fk, 0), xh8 = xsign(a.fk, 1);
  float r8[4], b8[4], fr8[4], fb8[4];
  auto bar64 = [&]() { asm volatile("bar.sync 1, 64;" ::: "memory"); };
  auto sweep8 = [&](float (&o)[4], const float (&n)[4], const float (&f)[4], float* so, float* sn,
                    bool up) {
    float x[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const float hi = m < 3 ? n[m + 1 & 3] : xh8 != 0.f ? xh8 * o[3] : n[0];
      const float lo = m > 0 ? n[m - 1 & 3] : xl8 != 0.f ? xl8 * o[0] : n[3];
      x[m] = up ? hi : lo;
    }
    relax4<PER>(o, n, x, f, sn, so, rw8, a.cu, a.cs, a.cf[0]);
    st4(so + own8, o);
    bar64();
  };
  auto smooth8 = [&](int steps, bool red0) {
    for (int q = 0; q < steps; ++q) {
      if (q > 0 || !red0) sweep8(r8, b8, fr8, cR, cB, e8);
      sweep8(b8, r8, fb8, cB, cR, !e8);
    }
  };
  for (int cyc = 0; cyc < a.cycles; ++cyc) {
    smooth16(a.pre, cyc == 0 && a.zero_guess);
    {  // restrict to 8^3 (four lanes hold a block's rows)
      float od[4], ev[4], xl[4], xr[4], d[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        od[m] = e ? r[m] : b[m];
        ev[m] = e ? b[m] : r[m];
      }
      float l = __shfl_xor_sync(0xffffffffu, od[3], 1), u = __shfl_xor_sync(0xffffffffu, ev[0], 1);
      if (!PER) {
        if (wl != 0.f) l = wl * ev[0];
        if (wh != 0.f) u = wh * od[3];
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        xl[m] = m > 0 ? od[m - 1 & 3] : l;
        xr[m] = m < 3 ? ev[m + 1 & 3] : u;
      }
      pair_defects<PER>(d, r, b, xl, xr, fr, fb, sR, sB, rw, a.ih2[1]);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        d[m] += __shfl_xor_sync(0xffffffffu, d[m], 2);
        d[m] += __shfl_xor_sync(0xffffffffu, d[m], 4);
        d[m] *= 0.125f;
      }
      if (!j0 && !k0) {  // cells 4 h .. 4 h + 3 of coarse row (J, K)
        const int o = K * S8 + J * 4 + 2 * h;
        const bool ec = (J + K) & 1;
        *reinterpret_cast<float2*>(cfR + o) = ec ? make_float2(d[1], d[3]) : make_float2(d[0], d[2]);
        *reinterpret_cast<float2*>(cfB + o) = ec ? make_float2(d[0], d[2]) : make_float2(d[1], d[3]);
      }
    }
    __syncthreads();
    if (t < 64) {
      const float4 x = ld4(cfR + own8), y = ld4(cfB + own8);
      fr8[0] = x.x; fr8[1] = x.y; fr8[2] = x.z; fr8[3] = x.w;
      fb8[0] = y.x; fb8[1] = y.y; fb8[2] = y.z; fb8[3] = y.w;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        r8[m] = a.pre > 0 ? a.cf[0] * fr8[m] : 0.f;
        b8[m] = 0.f;
      }
      st4(cR + own8, r8);
      st4(cB + own8, b8);
      bar64();
      smooth8(a.pre, true);
      float od[4], ev[4], xl[4], xr[4], d[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        od[m] = e8 ? r8[m] : b8[m];
        ev[m] = e8 ? b8[m] : r8[m];
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        xl[m] = m > 0 ? od[m - 1 & 3] : xl8 != 0.f ? xl8 * ev[0] : od[3];
        xr[m] = m < 3 ? ev[m + 1 & 3] : xh8 != 0.f ? xh8 * od[3] : ev[0];
      }
      pair_defects<PER>(d, r8, b8, xl, xr, fr8, fb8, cR, cB, rw8, a.ih2[0]);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        d[m] += __shfl_xor_sync(0xffffffffu, d[m], 1);
        d[m] += __shfl_xor_sync(0xffffffffu, d[m], 2);
        d[m] *= 0.125f;
      }
      if (!i8j && !i8k) st4(f4 + (K8 * 4 + J8) * 4, d);
    }
    __syncthreads();
    {  // the cycle of the levels from 4^3 down: eight lanes per row of the matrix
      const float4 x = ld4(f4 + 8 * (t & 7)), y = ld4(f4 + 8 * (t & 7) + 4);
      float v = (md[0] * x.x + md[1] * x.y) + (md[2] * x.z + md[3] * x.w);
      v += (md[4] * y.x + md[5] * y.y) + (md[6] * y.z + md[7] * y.w);
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      if ((t & 7) == 0) u4[t >> 3] = v;
    }
    __syncthreads();
    if (t < 64) {
      const Parents p = parents_of<4, PER>(a.fk, j8, k8, 4, 16);
      float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 c = ld4(u4 + p.o[q]);
        v[0] = fmaf(p.w[q], c.x, v[0]);
        v[1] = fmaf(p.w[q], c.y, v[1]);
        v[2] = fmaf(p.w[q], c.z, v[2]);
        v[3] = fmaf(p.w[q], c.w, v[3]);
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float lo = m > 0 ? v[m - 1 & 3] : xl8 != 0.f ? xl8 * v[0] : v[3];
        const float hi = m < 3 ? v[m + 1 & 3] : xh8 != 0.f ? xh8 * v[3] : v[0];
        const float ev = (3.f * v[m] + lo) * 0.015625f, od = (3.f * v[m] + hi) * 0.015625f;
        r8[m] += e8 ? od : ev;
        b8[m] += e8 ? ev : od;
      }
      st4(cR + own8, r8);
      st4(cB + own8, b8);
      bar64();
      smooth8(a.post, false);
      float n0[4], n1[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        (m < 2 ? n0 : n1)[2 * m & 3] = e8 ? b8[m] : r8[m];
        (m < 2 ? n0 : n1)[(2 * m & 3) + 1] = e8 ? r8[m] : b8[m];
      }
      st4(nat + (k8 * 8 + j8) * 8, n0);
      st4(nat + (k8 * 8 + j8) * 8 + 4, n1);
    }
    __syncthreads();
    {
      const Parents p = parents_of<8, PER>(a.fk, j, k, 8, 64);
      float v[8] = {};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 x = ld4(nat + p.o[q]), y = ld4(nat + p.o[q] + 4);
        const float w[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = fmaf(p.w[q], w[i], v[i]);
      }
      const float sl = xsign(a.fk, 0), sh = xsign(a.fk, 1);
      const float lo0 = h ? v[3] : sl != 0.f ? sl * v[0] : v[7];
      const float hi3 = h ? (sh != 0.f ? sh * v[7] : v[0]) : v[4];
      float c[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) c[m] = h ? v[m + 4] : v[m];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float lo = m > 0 ? c[m - 1 & 3] : lo0, hi = m < 3 ? c[m + 1 & 3] : hi3;
        const float ev = (3.f * c[m] + lo) * 0.015625f, od = (3.f * c[m] + hi) * 0.015625f;
        r[m] += e ? od : ev;
        b[m] += e ? ev : od;
      }
    }
    st4(sR + own, r);
    st4(sB + own, b);
    __syncthreads();
    smooth16(a.post, false);
  }
  float4 lo, hi;
  lo = e ? make_float4(b[0], r[0], b[1], r[1]) : make_float4(r[0], b[0], r[1], b[1]);
  hi = e ? make_float4(b[2], r[2], b[3], r[3]) : make_float4(r[2], b[2], r[3], b[3]);
  *reinterpret_cast<float4*>(a.u + g) = lo;
  *reinterpret_cast<float4*>(a.u + g + 4) = hi;
}

int log2i(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

// Kind of each face of a rule's homogeneous counterpart, 2 bits per face.
int face_kinds(const Bc& bc) {
  int fk = 0;
  for (int q = 0; q < 6; ++q) {
    int kind = face_kind(bc, q);
    if (kind == BC_OPEN) kind = BC_FIXED;
    fk |= kind << (2 * q);
  }
  return fk;
}

int swap_yz_kinds(int fk) { return (fk & 0x00f) | ((fk & 0x0f0) << 4) | ((fk & 0xf00) >> 4); }

constexpr int kCluster = 8;
// Most values (of T) a CTA holds: the cells of all its levels' u and f.
constexpr int kMaxValues = 26 * 1024;

// Shared-memory plan of levels 0 .. top: whether each is cut into slabs and
// where it lies.  Returns the values of T needed, or -1 where some level does
// not fit.
template <typename T>
int plan(const Grid* g, int top, bool one_cta, Level<T>* lev, bool swap) {
  int off = 0;
  for (int l = 0; l <= top; ++l) {
    const int ny = swap ? g[l].nz : g[l].ny, nz = swap ? g[l].ny : g[l].nz;
    const int plane = g[l].nx * ny;
    const bool whole = one_cta || (sizeof(T) == 4 && plane * nz <= 4096);
    const int dist = !whole && nz >= 2 * kCluster;
    if (!dist && plane * nz > 4096) return -1;
    if (l > 0 && g[l].nx < 2) return -1;
    const int planes = dist ? nz / kCluster : nz;
    if (lev) {
      lev[l].lx = log2i(g[l].nx);
      lev[l].ly = log2i(ny);
      lev[l].lz = log2i(nz);
      lev[l].dist = dist;
    }
    if (dist) off += plane;  // halo plane below
    if (lev) lev[l].u = off;
    off += planes * plane + (dist ? plane : 0);
    if (lev) lev[l].f = off;
    off += planes * plane;
  }
  return off <= kMaxValues ? off : -1;
}

template <typename T, bool PER, int MODE>
cudaError_t launch_mode(const cudaLaunchConfig_t& cfg, const CoarseArgs<T>& a) {
  static std::atomic<int> configured[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev].load()) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_coarse<T, PER, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kMaxValues * (int)sizeof(T));
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev].store(1);
  }
  return cudaLaunchKernelEx(&cfg, k_coarse<T, PER, MODE>, a);
}

// y and z change places when that cuts a level into slabs that would not be.
bool swap_for(const Grid& top) { return top.nz < 2 * kCluster && top.ny >= 2 * kCluster; }

}  // namespace

template <typename T>
int coarse_top(const Grid* g, int levels) {
  // FP64: up to 8192 cells (more would be bound by the cluster's FP64 units);
  // FP32: levels the fused legs do not take, up to what the cluster holds
  int t = 0;
  for (int l = 1; l < levels && l < kCoarseLevels; ++l) {
    const bool legs = g[l].nx >= 32 && g[l].ny >= 32 && g[l].nz >= 32;
    if (sizeof(T) == 4 ? legs || g[l].cells() > 32768 : g[l].cells() > 8192) break;
    if (plan<T>(g, l, false, nullptr, swap_for(g[l])) < 0) break;
    t = l;
  }
  return t;
}

template <typename T>
int coarse_fmg_top(const Grid* g, int levels) {
  int t = 0;
  for (int l = 1; l < levels && l < kCoarseLevels; ++l) {
    if (g[l].cells() > 1024 || plan<T>(g, l, true, nullptr, false) < 0) break;
    t = l;
  }
  return t;
}

int coarse_dense_level(const Grid* g, int levels) {
  for (int l = 1; l < levels && l < kCoarseLevels; ++l)
    if (g[l].cells() == kDense) return l;
  return 0;
}

template <typename T>
cudaError_t launch_coarse(const CoarseCall<T>& q, cudaStream_t s) {
  const int top = q.top;
  if (top < 1 || top >= kCoarseLevels) return cudaErrorInvalidValue;
  const Grid* g = q.g;
  const double* h = q.h;
  if constexpr (sizeof(T) == 4) {
    // (the FP32 path's rules are homogeneous)
    const Bc& b = q.bc[top];
    const bool plain = b.kind != BC_OPEN && (b.kind != BC_FIXED || b.value == 0.0) &&
                       (b.kind != BC_MIXED || !b.faces);
    if (q.mode == COARSE_CYCLES && plain && q.dense && g[top].nx == 16 && g[top].ny == 16 &&
        g[top].nz == 16 && (((uintptr_t)q.u | (uintptr_t)q.f) & 15u) == 0) {
      CubeArgs a{};
      a.u = q.u;
      a.f = q.f;
      a.dense = q.dense;
      a.cu = (float)(1.0 - q.omega);
      a.cs = (float)(q.omega / 6.0);
      for (int l = 0; l < 2; ++l) {
        const double hl = h[top - 1 + l];
        a.cf[l] = (float)(-q.omega * hl * hl / 6.0);
        a.ih2[l] = (float)(1.0 / (hl * hl));
      }
      a.fk_top = face_kinds(b);
      a.fk = face_kinds(q.hom);
      a.pre = q.pre;
      a.post = q.post;
      a.cycles = q.cycles;
      a.zero_guess = q.zero_guess ? 1 : 0;
      ++g_launches;
      if (a.fk_top == 0 && a.fk == 0) launch_after(k_cube16<true>, 1, kCubeThreads, 0, s, a);
      else launch_after(k_cube16<false>, 1, kCubeThreads, 0, s, a);
      return cudaGetLastError();
    }
  }
  const bool one_cta = q.mode != COARSE_CYCLES;
  CoarseArgs<T> a{};
  a.swap_yz = !one_cta && swap_for(g[top]);
  const int values = plan<T>(g, top, one_cta, a.lev, a.swap_yz);
  if (values < 0) return cudaErrorInvalidValue;
  for (int l = 0; l <= top; ++l) {
    a.lev[l].cf = (T)(-q.omega * h[l] * h[l] / 6.0);
    a.lev[l].ih2 = (T)(1.0 / (h[l] * h[l]));
    a.h[l] = h[l];
    a.bc[l] = q.mode == COARSE_FMG || l == top ? q.bc[l] : q.hom;
  }
  a.u_top = q.u;
  a.f_top = q.f;
  a.sy = g[top].nx;
  a.sz = (long long)g[top].nx * g[top].ny;
  if (a.swap_yz) {
    const long long t = a.sy;
    a.sy = a.sz;
    a.sz = t;
  }
  a.cu = (T)(1.0 - q.omega);
  a.cs = (T)(q.omega / 6.0);
  a.cf0 = (T)(-h[0] * h[0] / 6.0);
  a.top = top;
  a.pre = q.pre;
  a.post = q.post;
  a.cycles = q.cycles;
  a.zero_guess = q.zero_guess ? 1 : 0;
  a.fk_top = face_kinds(q.bc[top]);
  a.fk = face_kinds(q.hom);
  a.nmax0 = g[0].nx > g[0].ny ? g[0].nx : g[0].ny;
  if (g[0].nz > a.nmax0) a.nmax0 = g[0].nz;
  if (a.swap_yz) {
    a.fk_top = swap_yz_kinds(a.fk_top);
    a.fk = swap_yz_kinds(a.fk);
  }
  // the matrix is in the order of the level's own axes
  if (q.dense && q.mode != COARSE_BASIS && !a.swap_yz) {
    a.dense = q.dense;
    a.dense_level = coarse_dense_level(g, top + 1);
  }
  const bool per = a.fk_top == 0 && a.fk == 0;  // BC_PERIODIC on every face
  bool any = false;
  for (int l = 0; l <= top; ++l) any = any || a.lev[l].dist;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[2];
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = any ? kCluster : 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(q.mode == COARSE_BASIS ? kDense : any ? kCluster : 1);
  cfg.blockDim = dim3(kThreads<T>);
  cfg.dynamicSmemBytes = (size_t)values * sizeof(T);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  ++g_launches;
  if (q.mode == COARSE_FMG)
    return per ? launch_mode<T, true, COARSE_FMG>(cfg, a) : launch_mode<T, false, COARSE_FMG>(cfg, a);
  if (q.mode == COARSE_BASIS)
    return per ? launch_mode<T, true, COARSE_BASIS>(cfg, a)
               : launch_mode<T, false, COARSE_BASIS>(cfg, a);
  return per ? launch_mode<T, true, COARSE_CYCLES>(cfg, a)
             : launch_mode<T, false, COARSE_CYCLES>(cfg, a);
}

#define MG_INSTANTIATE(T)                       \
  template int coarse_top<T>(const Grid*, int); \
  template int coarse_fmg_top<T>(const Grid*, int); \
  template cudaError_t launch_coarse<T>(const CoarseCall<T>&, cudaStream_t);

MG_INSTANTIATE(float)
MG_INSTANTIATE(double)

}  // namespace mg
