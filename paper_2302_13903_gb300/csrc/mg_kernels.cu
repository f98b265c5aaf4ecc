// mg_kernels.cu -- per-level multigrid kernels for sm_103a (FP64 and FP32).
//
// Layout: every level is an nx*ny*nz array of active cells, z-major, x
// fastest; there are no ghost cells in memory.  A neighbour outside the level
// is synthesised from the boundary rule at load time (Sec. 2.3.6): periodic
// wraps, zero gradient copies the adjacent cell, fixed / open give
// 2 b - (adjacent cell) with b the value on the face.  Where a stencil leaves
// the level along more than one axis (edges and corners of the 27-point
// prolongations) the face rule is applied along x, then y, then z.
//
// These are the straightforward kernels: one thread per output cell (or per
// coarse cell for the fused defect + restriction), grid-stride loops over the
// bodies in mg_device.cuh, and deterministic two-stage reductions.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "mg_convert.cuh"
#include "mg_device.cuh"
#include "mg_internal.h"

namespace mg {

thread_local long long g_launches = 0;

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Deterministic block sum (blockDim.x == kThreads); result valid in thread 0.
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double ws[kThreads / 32];
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) ws[w] = v;
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    r = lane < kThreads / 32 ? ws[lane] : 0.0;
    r = warp_sum(r);
  }
  __syncthreads();
  return r;
}

int grid_for(long long work) {
  long long b = (work + kThreads - 1) / kThreads;
  if (b < 1) b = 1;
  if (b > sm_count() * 64LL) b = sm_count() * 64LL;
  return (int)b;
}

// Threads per block of a level kernel with `work` items: 256, or 64 where blocks
// of 256 would leave SMs, and with them FP64 units, without one (32^3: 32
// blocks on 152 SMs).  FP64 solves with 64 there and with 256 everywhere (GB300, us):
// 32^3 fixed 1098, 1148; 64^3 periodic 964, 991; 128^3 1493, 1532; 256^3 4832, 4889.
int threads_for(long long work) { return work < 256LL * sm_count() ? 64 : kThreads; }
int blocks_for(long long work) {
  const int t = threads_for(work);
  long long b = (work + t - 1) / t;
  if (b > sm_count() * 64LL) b = sm_count() * 64LL;
  return b < 1 ? 1 : (int)b;
}

// ---------------------------------------------------------------------------
// Level kernels for even sizes.  In FP64 an SM issues two operations per clock,
// so what counts is the number of FP64 operations per cell and that no warp
// runs two versions of them: a lane at a face selects what it loads (the
// periodic image, or the ghost of Sec. 2.3.6) and then takes the same path as
// the others.  A thread has a patch of 2 x 2 cells in (x, y), because the two
// cells of one colour in it share the sum of the two others:
//   j+1:  Y B      A and B of one colour: A's x and y neighbours inside the
//   j  :  A X      patch are X and Y, and so are B's (or mirrored in x).

// The neighbour of a cell across face q: ghost from the rule.
template <typename T>
__device__ __noinline__ T face_ghost(const T* u, T self, int q, int i, int j, int k, const Grid g,
                                     const Bc bc) {
  const int kind = face_kind(bc, q);
  if (kind == BC_PERIODIC) {
    const int hi = q & 1;
    if (q < 2) i = hi ? 0 : g.nx - 1;
    else if (q < 4) j = hi ? 0 : g.ny - 1;
    else k = hi ? 0 : g.nz - 1;
    return u[dev::at(g, i, j, k)];
  }
  if (kind == BC_ZEROGRAD) return self;
  const T b = (T)dev::face_value(bc, g, q, (q < 2 ? j : i) + 1, (q < 4 ? k : j) + 1);
  return T(2) * b - self;
}

// Neighbours of cell c = (i, j, k) along one axis: lower (q even) or upper.
template <typename T, bool PER>
struct Around {
  const T* u;
  const Grid& g;
  const Bc& bc;
  __device__ __forceinline__ T x(size_t c, int i, int j, int k, int hi) const {
    const bool in = hi ? i < g.nx - 1 : i > 0;
    if (PER) return u[in ? (hi ? c + 1 : c - 1) : (hi ? c + 1 - g.nx : c + g.nx - 1)];
    return in ? u[hi ? c + 1 : c - 1] : face_ghost(u, u[c], hi, i, j, k, g, bc);
  }
  __device__ __forceinline__ T y(size_t c, int i, int j, int k, int hi) const {
    const size_t sy = (size_t)g.nx, w = sy * (g.ny - 1);
    const bool in = hi ? j < g.ny - 1 : j > 0;
    if (PER) return u[in ? (hi ? c + sy : c - sy) : (hi ? c - w : c + w)];
    return in ? u[hi ? c + sy : c - sy] : face_ghost(u, u[c], 2 + hi, i, j, k, g, bc);
  }
  __device__ __forceinline__ T z(size_t c, int i, int j, int k, int hi) const {
    const size_t sz = (size_t)g.nx * g.ny, w = sz * (g.nz - 1);
    const bool in = hi ? k < g.nz - 1 : k > 0;
    if (PER) return u[in ? (hi ? c + sz : c - sz) : (hi ? c - w : c + w)];
    return in ? u[hi ? c + sz : c - sz] : face_ghost(u, u[c], 4 + hi, i, j, k, g, bc);
  }
  // Neighbour sums of the patch's two cells of one colour: cell A of row j is
  // 2 m + e, cell B of row j + 1 is 2 m + 1 - e (nine additions for both).
  __device__ __forceinline__ void sums(int m, int j, int k, int e, size_t& ca, size_t& cb, T& sa,
                                       T& sb) const {
    const int ia = 2 * m + e, ib = 2 * m + 1 - e;
    ca = dev::at(g, ia, j, k);
    cb = dev::at(g, ib, j + 1, k);
    const T p = u[dev::at(g, ib, j, k)] + u[dev::at(g, ia, j + 1, k)];
    sa = (p + (x(ca, ia, j, k, e) + y(ca, ia, j, k, 0))) + (z(ca, ia, j, k, 0) + z(ca, ia, j, k, 1));
    sb = (p + (x(cb, ib, j + 1, k, 1 - e) + y(cb, ib, j + 1, k, 1))) +
         (z(cb, ib, j + 1, k, 0) + z(cb, ib, j + 1, k, 1));
  }
};

// One colour of SMOOTH: 7.5 operations per updated cell.
template <typename T, bool PER>
__global__ void __launch_bounds__(kThreads) k_sor_patch(T* u, const T* f, Grid g, Bc bc, T cu, T cs,
                                                        T cf, int colour) {
  dev::after_previous();
  const int hx = g.nx >> 1, hy = g.ny >> 1;
  const long long total = (long long)hx * hy * g.nz;
  const dev::Split sp(hx, hy);
  const Around<T, PER> n{u, g, bc};
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int m, jj, k;
    sp(t, m, jj, k);
    size_t ca, cb;
    T sa, sb;
    n.sums(m, 2 * jj, k, (k + colour) & 1, ca, cb, sa, sb);
    const T va = cs * sa + (cu * u[ca] + cf * f[ca]);
    const T vb = cs * sb + (cu * u[cb] + cf * f[cb]);
    u[ca] = va;
    u[cb] = vb;
  }
}

// Partial sums of d^2, d = f - (sum_nb - 6 u) / h^2: 7.5 operations per cell.
// R32: also r32 = scale d, narrowed by integer arithmetic.
template <typename T, bool PER, bool R32>
__global__ void __launch_bounds__(kThreads) k_defect_norm(const T* u, const T* f, Grid g, Bc bc,
                                                          T inv_h2, double* partials, float* r32,
                                                          double scale) {
  dev::after_previous();
  const int hx = g.nx >> 1, hy = g.ny >> 1;
  const long long total = (long long)hx * hy * g.nz;
  const dev::Split sp(hx, hy);
  const Around<T, PER> n{u, g, bc};
  double acc = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    int m, jj, k;
    sp(t, m, jj, k);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      size_t ca, cb;
      T sa, sb;
      n.sums(m, 2 * jj, k, e, ca, cb, sa, sb);
      const T da = f[ca] - (sa - T(6) * u[ca]) * inv_h2;
      const T db = f[cb] - (sb - T(6) * u[cb]) * inv_h2;
      acc += (double)da * (double)da;
      acc += (double)db * (double)db;
      if (R32) {
        r32[ca] = cvt::d2f_rn((double)da * scale);
        r32[cb] = cvt::d2f_rn((double)db * scale);
      }
    }
  }
  const double b = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

// Defect of the eight children of each coarse cell, averaged (Algorithm 1,
// steps 2-3).  Summed over the block, the neighbour sums are three times the
// sum of the eight cells (each has three neighbours among them) plus the 24
// cells around it: 40 operations per block where a defect per cell takes 72.
// Two neighbouring lanes share a block, a plane each.
template <typename T, bool PER>
__global__ void __launch_bounds__(kThreads) k_defect_restrict_block(const T* u, const T* f, T* fc,
                                                                    Grid g, Bc bc, T inv_h2) {
  dev::after_previous();
  const Grid gc{g.nx / 2, g.ny / 2, g.nz / 2};
  const long long work = 2 * gc.cells();
  const dev::Split sp(gc.nx, gc.ny);
  const Around<T, PER> n{u, g, bc};
  for (long long t0 = blockIdx.x * (long long)blockDim.x; t0 < work;
       t0 += (long long)gridDim.x * blockDim.x) {
    const long long t = t0 + threadIdx.x;
    const bool live = t < work;
    const int d = (int)(t & 1);
    int I, J, K;
    sp(live ? t >> 1 : 0, I, J, K);
    const int i = 2 * I, j = 2 * J, k = 2 * K + d;
    const size_t c = dev::at(g, i, j, k), cy = c + g.nx;
    const T own = (u[c] + u[c + 1]) + (u[cy] + u[cy + 1]);
    const T fs = (f[c] + f[c + 1]) + (f[cy] + f[cy + 1]);
    const T ox = (n.x(c, i, j, k, 0) + n.x(cy, i, j + 1, k, 0)) +
                 (n.x(c + 1, i + 1, j, k, 1) + n.x(cy + 1, i + 1, j + 1, k, 1));
    const T oy = (n.y(c, i, j, k, 0) + n.y(c + 1, i + 1, j, k, 0)) +
                 (n.y(cy, i, j + 1, k, 1) + n.y(cy + 1, i + 1, j + 1, k, 1));
    const T oz = (n.z(c, i, j, k, d) + n.z(c + 1, i + 1, j, k, d)) +
                 (n.z(cy, i, j + 1, k, d) + n.z(cy + 1, i + 1, j + 1, k, d));
    T v = fs - inv_h2 * (((ox + oy) + oz) - T(3) * own);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    if (live && !d) fc[t >> 1] = v * T(0.125);
  }
}

// u += trilinear(uc) for a homogeneous coarse rule, over z-chunks of coarse
// columns: the (x, y) interpolation of a coarse plane is formed once and kept
// for the three pairs of fine planes that use it.  Interpolating 4 x by
// 3 b + a (one operation) leaves a factor of 64 to the last, fused with the
// addition to u: 26 operations per coarse cell and plane, where weights 1/4 and
// 3/4 take 35.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_prolong_add(const T* uc, T* uf, Grid gf, Bc bc, int cz,
                                                          long long items) {
  dev::after_previous();
  const Grid gc{gf.nx / 2, gf.ny / 2, gf.nz / 2};
  const dev::Split sp(gc.nx, gc.ny);
  const size_t plane = (size_t)gf.nx * gf.ny, planec = (size_t)gc.nx * gc.ny;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < items;
       t += (long long)gridDim.x * blockDim.x) {
    int I, J, ch;
    sp(t, I, J, ch);
    const int K0 = ch * cz, K1 = min(K0 + cz, gc.nz);
    // offset of the coarse neighbour on each side and whether it enters with
    // a minus sign (the cell itself stands in for it at a wall)
    int ox[3] = {0, 0, 0}, oy[3] = {0, 0, 0};
    unsigned neg = 0;  // bits 0 x-, 1 x+, 2 y-, 3 y+
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
      const bool inx = hi ? I < gc.nx - 1 : I > 0, iny = hi ? J < gc.ny - 1 : J > 0;
      const int kx = face_kind(bc, hi), ky = face_kind(bc, 2 + hi);
      ox[2 * hi] = inx ? 2 * hi - 1 : kx == BC_PERIODIC ? (1 - 2 * hi) * (gc.nx - 1) : 0;
      oy[2 * hi] = (iny ? 2 * hi - 1 : ky == BC_PERIODIC ? (1 - 2 * hi) * (gc.ny - 1) : 0) * gc.nx;
      if (!inx && kx == BC_FIXED) neg |= 1u << hi;
      if (!iny && ky == BC_FIXED) neg |= 4u << hi;
    }
    auto xy = [&](int K, T out[2][2]) {
      bool nz = false;
      if (K < 0 || K >= gc.nz) {
        const int kz = face_kind(bc, K < 0 ? 4 : 5);
        nz = kz == BC_FIXED;
        K = (K < 0) == (kz == BC_PERIODIC) ? gc.nz - 1 : 0;
      }
      const T* p = uc + (size_t)K * planec + (size_t)J * gc.nx + I;
      T vx[3][2];
#pragma unroll
      for (int y = 0; y < 3; ++y) {
        T v[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          v[x] = p[ox[x] + oy[y]];
          const bool n = (x != 1 && (neg >> (x >> 1) & 1)) != (y != 1 && (neg >> (2 + (y >> 1)) & 1));
          if (n != nz) v[x] = -v[x];
        }
        vx[y][0] = T(3) * v[1] + v[0];
        vx[y][1] = T(3) * v[1] + v[2];
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        out[0][x] = T(3) * vx[1][x] + vx[0][x];
        out[1][x] = T(3) * vx[1][x] + vx[2][x];
      }
    };
    T pm[2][2], p0[2][2], pp[2][2];
    xy(K0 - 1, pm);
    xy(K0, p0);
    for (int K = K0; K < K1; ++K) {
      xy(K + 1, pp);
#pragma unroll
      for (int y = 0; y < 2; ++y)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const size_t q = dev::at(gf, 2 * I + x, 2 * J + y, 2 * K);
          uf[q] = T(1.0 / 64) * (T(3) * p0[y][x] + pm[y][x]) + uf[q];
          uf[q + plane] = T(1.0 / 64) * (T(3) * p0[y][x] + pp[y][x]) + uf[q + plane];
          pm[y][x] = p0[y][x];
          p0[y][x] = pp[y][x];
        }
    }
  }
}

bool even_sizes(const Grid& g) { return g.nx % 2 == 0 && g.ny % 2 == 0 && g.nz % 2 == 0; }
bool homogeneous_rule(const Bc& bc) {
  return bc.kind == BC_PERIODIC || bc.kind == BC_ZEROGRAD ||
         (bc.kind == BC_FIXED && bc.value == 0.0) || (bc.kind == BC_MIXED && !bc.faces);
}

// ---------------------------------------------------------------------------
// d = f - (sum_nb - 6u) / h^2; optional store and partial sums of d^2.
template <typename T>
__global__ void k_defect(const T* u, const T* f, T* __restrict__ d,
                         Grid g, Bc bc, T inv_h2, double* __restrict__ partials) {
  dev::after_previous();
  const long long total = g.cells();
  double acc = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % g.nx);
    const long long r = t / g.nx;
    const int j = (int)(r % g.ny), k = (int)(r / g.ny);
    const T s = dev::neighbour_sum(u, i, j, k, g, bc);
    const T dv = f[t] - (s - T(6) * u[t]) * inv_h2;
    if (d) d[t] = dv;
    acc += (double)dv * (double)dv;
  }
  if (partials) {
    const double b = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = b;
  }
}

template <typename T>
__global__ void k_sor(T* u, const T* f, Grid g, Bc bc, T cu, T cs, T cf, int colour) {
  dev::after_previous();
  dev::sor_range(u, f, g, bc, cu, cs, cf, colour, blockIdx.x * (long long)blockDim.x + threadIdx.x,
                 (long long)gridDim.x * blockDim.x);
}

template <typename T>
__global__ void k_sor_red_zero(T* u, const T* f, Grid g, T cf) {
  dev::after_previous();
  dev::sor_red_zero_range(u, f, g, cf, blockIdx.x * (long long)blockDim.x + threadIdx.x,
                          (long long)gridDim.x * blockDim.x);
}

template <typename T>
__global__ void k_defect_restrict(const T* u, const T* f, T* fc, Grid g, Bc bc, T inv_h2) {
  dev::after_previous();
  dev::defect_restrict_range(u, f, fc, g, bc, inv_h2,
                             blockIdx.x * (long long)blockDim.x + threadIdx.x,
                             (long long)gridDim.x * blockDim.x);
}

template <typename T>
__global__ void k_restrict(const T* uf, T* uc, Grid gf) {
  dev::after_previous();
  dev::restrict_range(uf, uc, gf, blockIdx.x * (long long)blockDim.x + threadIdx.x,
                      (long long)gridDim.x * blockDim.x);
}

template <typename T, bool HIGH>
__global__ void k_prolong(const T* uc, T* uf, Grid gf, Bc bc, int add, int cz, long long items) {
  dev::after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < items;
       t += (long long)gridDim.x * blockDim.x)
    dev::prolong_zchunk<T, HIGH>(uc, uf, gf, bc, add, t, cz);
}

template <typename T>
__global__ void k_coarsest(const T* f, T* u, double h, Bc bc, bool keep) {
  dev::after_previous();
  if (threadIdx.x == 0 && blockIdx.x == 0) dev::coarsest_one(f, u, h, bc, keep);
}

template <typename T>
__global__ void k_fill(T* __restrict__ u, long long n, T v) {
  dev::after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    u[t] = v;
}

__global__ void k_add_const(double* __restrict__ u, long long n, double v) {
  dev::after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    u[t] += v;
}

// f = 4 pi G rho and partial sums of f, or of f^2 (SQ).
template <bool SQ>
__global__ void k_source(const double* rho, double* __restrict__ f, long long n,
                         double four_pi_G, double* __restrict__ partials) {
  dev::after_previous();
  double acc = 0.0;
#pragma unroll 4
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const double v = four_pi_G * rho[t];
    f[t] = v;
    acc = SQ ? fma(v, v, acc) : acc + v;
  }
  const double b = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

template <typename T>
__global__ void k_sum(const T* a, long long n, int squares,
                      double* __restrict__ partials) {
  dev::after_previous();
  double acc = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const double v = (double)a[t];
    acc += squares ? v * v : v;
  }
  const double b = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

// flag: also *flag, as a double, into out[1].
__global__ void k_finish_sum(const double* partials, int nb, double* __restrict__ out,
                             const int* flag) {
  dev::after_previous();
  double acc = 0.0;
#pragma unroll 8
  for (int t = threadIdx.x; t < nb; t += kThreads) acc += partials[t];
  const double b = block_sum(acc);
  if (threadIdx.x == 0) {
    out[0] = b;
    if (flag) out[1] = (double)*flag;
  }
}

// a -= total[0] / n (the total was formed on the device in a fixed order);
// SQ: partial sums of the new a^2.
template <bool SQ>
__global__ void k_subtract_mean(double* __restrict__ a, long long n, const double* total,
                                double* __restrict__ partials) {
  dev::after_previous();
  const double mean = total[0] / (double)n;
  double acc = 0.0;
#pragma unroll 4
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const double v = a[t] - mean;
    a[t] = v;
    if (SQ) acc = fma(v, v, acc);
  }
  if (SQ) {
    const double b = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = b;
  }
}

__global__ void k_scale_to_f32(const double* a, float* __restrict__ b, long long n,
                               double scale) {
  dev::after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    b[t] = (float)(scale * a[t]);
}

__global__ void k_correct(double* __restrict__ u, const float* e, long long n,
                          double inv_scale) {
  dev::after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    u[t] += inv_scale * (double)e[t];
}

// Algorithm 3 step 5 on a coarse level: f += L ur (the restricted potential's
// Laplacian with the level's own rule) and the start value u = ur.
__global__ void k_fas_rhs(const double* ur, double* __restrict__ f,
                          double* __restrict__ u, Grid g, Bc bc, double inv_h2) {
  dev::after_previous();
  const long long total = g.cells();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % g.nx);
    const long long r = t / g.nx;
    const int j = (int)(r % g.ny), k = (int)(r / g.ny);
    const double s = dev::neighbour_sum(ur, i, j, k, g, bc);
    f[t] += (s - 6.0 * ur[t]) * inv_h2;
    u[t] = ur[t];
  }
}

// Algorithm 3 step 7: u -= ur (the coarse-grid correction).
__global__ void k_sub(double* __restrict__ u, const double* ur, long long n) {
  dev::after_previous();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    u[t] -= ur[t];
}

// g = -grad phi at cell centres (Sec. 3.2.3): per axis the average of the two
// face accelerations -(phi_{i+1} - phi_i) / h and -(phi_i - phi_{i-1}) / h,
// neighbours outside the level from the rule; g = [g_x | g_y | g_z].
__global__ void k_gravity(const double* u, double* __restrict__ g, Grid gr, Bc bc,
                          double h) {
  dev::after_previous();
  const long long total = gr.cells();
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % gr.nx);
    const long long r = t / gr.nx;
    const int j = (int)(r % gr.ny), k = (int)(r / gr.ny);
    const double c = u[t];
    const double xl = -(c - dev::fetch(u, i - 1, j, k, gr, bc)) / h;
    const double xr = -(dev::fetch(u, i + 1, j, k, gr, bc) - c) / h;
    const double yl = -(c - dev::fetch(u, i, j - 1, k, gr, bc)) / h;
    const double yr = -(dev::fetch(u, i, j + 1, k, gr, bc) - c) / h;
    const double zl = -(c - dev::fetch(u, i, j, k - 1, gr, bc)) / h;
    const double zr = -(dev::fetch(u, i, j, k + 1, gr, bc) - c) / h;
    g[t] = 0.5 * (xl + xr);
    g[total + t] = 0.5 * (yl + yr);
    g[2 * total + t] = 0.5 * (zl + zr);
  }
}

}  // namespace

int sm_count() {
  static std::atomic<int> cached[64];  // zero-initialised (static storage)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return 152;
  }
  int n = cached[dev].load();
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
      cudaGetLastError();
      n = 152;
    }
    cached[dev].store(n);
  }
  return n;
}

int reduce_blocks(long long n) {
  long long b = (n + kThreads * 4 - 1) / (kThreads * 4);
  if (b < 1) b = 1;
  if (b > kMaxReduceBlocks) b = kMaxReduceBlocks;
  return (int)b;
}

template <typename T>
cudaError_t launch_sor(T* u, const T* f, Grid g, double h, Bc bc, double omega, int colour,
                       cudaStream_t s) {
  const long long work = (long long)(g.nx / 2) * g.ny * g.nz;
  const T cu = (T)(1.0 - omega), cs = (T)(omega / 6.0), cf = (T)(-omega * h * h / 6.0);
  ++g_launches;
  if (g.nx % 2 == 0 && g.ny % 2 == 0) {
    if (bc.kind == BC_PERIODIC)
      launch_after(k_sor_patch<T, true>, blocks_for(work / 2), threads_for(work / 2), 0, s, u, f, g,
                   bc, cu, cs, cf, colour);
    else
      launch_after(k_sor_patch<T, false>, blocks_for(work / 2), threads_for(work / 2), 0, s, u, f,
                   g, bc, cu, cs, cf, colour);
  } else {
    launch_after(k_sor<T>, grid_for(work), kThreads, 0, s, u, f, g, bc, cu, cs, cf, colour);
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_sor_red_zero(T* u, const T* f, Grid g, double h, double omega,
                                cudaStream_t s) {
  ++g_launches;
  launch_after(k_sor_red_zero<T>, blocks_for(g.cells()), threads_for(g.cells()), 0, s, u, f, g,
               (T)(-omega * h * h / 6.0));
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_defect(const T* u, const T* f, T* d, Grid g, double h, Bc bc, double* partials,
                          cudaStream_t s) {
  ++g_launches;
  const int nb = partials ? reduce_blocks(g.cells()) : grid_for(g.cells());
  if (partials && !d && g.nx % 2 == 0 && g.ny % 2 == 0) {
    const T ih2 = (T)(1.0 / (h * h));
    if (bc.kind == BC_PERIODIC)
      launch_after(k_defect_norm<T, true, false>, nb, kThreads, 0, s, u, f, g, bc, ih2, partials,
                   nullptr, 0.0);
    else
      launch_after(k_defect_norm<T, false, false>, nb, kThreads, 0, s, u, f, g, bc, ih2, partials,
                   nullptr, 0.0);
    return cudaGetLastError();
  }
  launch_after(k_defect<T>, nb, kThreads, 0, s, u, f, d, g, bc, (T)(1.0 / (h * h)), partials);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_defect_restrict(const T* u, const T* f, T* fc, Grid g, double h, Bc bc,
                                   cudaStream_t s) {
  ++g_launches;
  const T ih2 = (T)(1.0 / (h * h));
  if (!even_sizes(g))
    launch_after(k_defect_restrict<T>, grid_for(g.cells() / 8), kThreads, 0, s, u, f, fc, g, bc, ih2);
  else if (bc.kind == BC_PERIODIC)
    launch_after(k_defect_restrict_block<T, true>, blocks_for(g.cells() / 4),
                 threads_for(g.cells() / 4), 0, s, u, f, fc, g, bc, ih2);
  else
    launch_after(k_defect_restrict_block<T, false>, blocks_for(g.cells() / 4),
                 threads_for(g.cells() / 4), 0, s, u, f, fc, g, bc, ih2);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_restrict(const T* uf, T* uc, Grid gf, cudaStream_t s) {
  ++g_launches;
  launch_after(k_restrict<T>, grid_for(gf.cells() / 8), kThreads, 0, s, uf, uc, gf);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_prolong(const T* uc, T* uf, Grid gf, Bc bc_coarse, int high_order, int add,
                           cudaStream_t s) {
  ++g_launches;
  // z-chunks of coarse columns: 8 planes each while that leaves about 2^16
  // work items (three FP64 warps per scheduler), fewer on small levels.  With 2^18
  // FP64 solves took (GB300) 256^3 periodic 4853 us instead of 4832, fixed 7128
  // instead of 7090, the smaller ones the same
  const long long cols = (long long)(gf.nx / 2) * (gf.ny / 2);
  const int cnz = gf.nz / 2;
  int cz = 8;
  while (cz > 1 && cols * ((cnz + cz - 1) / cz) < (1LL << 16)) cz /= 2;
  const long long items = cols * ((cnz + cz - 1) / cz);
  if (!high_order && add && homogeneous_rule(bc_coarse))
    launch_after(k_prolong_add<T>, blocks_for(items), threads_for(items), 0, s, uc, uf, gf,
                 bc_coarse, cz, items);
  else if (high_order)
    launch_after(k_prolong<T, true>, blocks_for(items), threads_for(items), 0, s, uc, uf, gf,
                 bc_coarse, add, cz, items);
  else
    launch_after(k_prolong<T, false>, blocks_for(items), threads_for(items), 0, s, uc, uf, gf,
                 bc_coarse, add, cz, items);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_coarsest(const T* f, T* u, double h, Bc bc, cudaStream_t s, bool keep) {
  ++g_launches;
  launch_after(k_coarsest<T>, 1, 32, 0, s, f, u, h, bc, keep);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_fill(T* u, long long n, T v, cudaStream_t s) {
  ++g_launches;
  launch_after(k_fill<T>, grid_for(n), kThreads, 0, s, u, n, v);
  return cudaGetLastError();
}

cudaError_t launch_source(const double* rho, double* f, long long n, double four_pi_G, bool squares,
                          double* partials, cudaStream_t s) {
  ++g_launches;
  if (squares) launch_after(k_source<true>, reduce_blocks(n), kThreads, 0, s, rho, f, n, four_pi_G, partials);
  else launch_after(k_source<false>, reduce_blocks(n), kThreads, 0, s, rho, f, n, four_pi_G, partials);
  return cudaGetLastError();
}

cudaError_t launch_subtract_mean(double* a, long long n, double* partials, int nb,
                                 double* total_slot, bool squares, cudaStream_t s) {
  ++g_launches;
  launch_after(k_finish_sum, 1, kThreads, 0, s, partials, nb, total_slot, nullptr);
  ++g_launches;
  if (squares)
    launch_after(k_subtract_mean<true>, reduce_blocks(n), kThreads, 0, s, a, n, total_slot, partials);
  else
    launch_after(k_subtract_mean<false>, grid_for(n), kThreads, 0, s, a, n, total_slot, nullptr);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_sum(const T* a, long long n, int squares, double* partials, cudaStream_t s) {
  ++g_launches;
  launch_after(k_sum<T>, reduce_blocks(n), kThreads, 0, s, a, n, squares, partials);
  return cudaGetLastError();
}

cudaError_t launch_fas_rhs(const double* ur, double* f, double* u, Grid g, double h, Bc bc,
                           cudaStream_t s) {
  ++g_launches;
  launch_after(k_fas_rhs, grid_for(g.cells()), kThreads, 0, s, ur, f, u, g, bc, 1.0 / (h * h));
  return cudaGetLastError();
}

cudaError_t launch_sub(double* u, const double* ur, long long n, cudaStream_t s) {
  ++g_launches;
  launch_after(k_sub, grid_for(n), kThreads, 0, s, u, ur, n);
  return cudaGetLastError();
}

cudaError_t launch_gravity(const double* u, double* g, Grid gr, double h, Bc bc, cudaStream_t s) {
  ++g_launches;
  launch_after(k_gravity, grid_for(gr.cells()), kThreads, 0, s, u, g, gr, bc, h);
  return cudaGetLastError();
}

cudaError_t launch_finish_sum(const double* partials, int nb, double* out, cudaStream_t s,
                              const int* flag) {
  ++g_launches;
  launch_after(k_finish_sum, 1, kThreads, 0, s, partials, nb, out, flag);
  return cudaGetLastError();
}

cudaError_t launch_outer_residual(const double* u, const double* f, float* r32, Grid g, double h,
                                  Bc bc, double scale, double* partials, cudaStream_t s) {
  ++g_launches;
  if (g.nx % 2 || g.ny % 2) return cudaErrorInvalidValue;  // levels have sides 2^k >= 2
  auto kernel = bc.kind == BC_PERIODIC ? k_defect_norm<double, true, true>
                                       : k_defect_norm<double, false, true>;
  launch_after(kernel, reduce_blocks(g.cells()), kThreads, 0, s, u, f, g, bc, 1.0 / (h * h),
               partials, r32, scale);
  return cudaGetLastError();
}

cudaError_t launch_add_const(double* u, long long n, double v, cudaStream_t s) {
  ++g_launches;
  launch_after(k_add_const, grid_for(n), kThreads, 0, s, u, n, v);
  return cudaGetLastError();
}

cudaError_t launch_scale_to_f32(const double* a, float* b, long long n, double scale,
                               cudaStream_t s) {
  ++g_launches;
  launch_after(k_scale_to_f32, grid_for(n), kThreads, 0, s, a, b, n, scale);
  return cudaGetLastError();
}

cudaError_t launch_correct(double* u, const float* e32, long long n, double inv_scale,
                           cudaStream_t s) {
  ++g_launches;
  launch_after(k_correct, grid_for(n), kThreads, 0, s, u, e32, n, inv_scale);
  return cudaGetLastError();
}

#define MG_INSTANTIATE(T)                                                                        \
  template cudaError_t launch_sor<T>(T*, const T*, Grid, double, Bc, double, int, cudaStream_t); \
  template cudaError_t launch_sor_red_zero<T>(T*, const T*, Grid, double, double, cudaStream_t); \
  template cudaError_t launch_defect<T>(const T*, const T*, T*, Grid, double, Bc, double*,       \
                                        cudaStream_t);                                           \
  template cudaError_t launch_defect_restrict<T>(const T*, const T*, T*, Grid, double, Bc,       \
                                                 cudaStream_t);                                  \
  template cudaError_t launch_restrict<T>(const T*, T*, Grid, cudaStream_t);                     \
  template cudaError_t launch_prolong<T>(const T*, T*, Grid, Bc, int, int, cudaStream_t);        \
  template cudaError_t launch_coarsest<T>(const T*, T*, double, Bc, cudaStream_t, bool);         \
  template cudaError_t launch_fill<T>(T*, long long, T, cudaStream_t);                           \
  template cudaError_t launch_sum<T>(const T*, long long, int, double*, cudaStream_t);

MG_INSTANTIATE(float)
MG_INSTANTIATE(double)

}  // namespace mg
